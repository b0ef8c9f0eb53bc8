"""The work that users of this library have it do, as cases that can be timed and checked.

Each case goes through the package's public calls: moments of the density of states and
their reconstruction, many systems in one launch, 2D moments, the conductivities built
from them, the k-resolved spectral function, wave-packet evolution and the learned density.
``exact`` restates each of them in 64 bits with torch and numpy alone.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

import paper_1910_05194_gb300 as kite

DEV = "cuda:0"
T_HOP = {"honeycomb": -2.7, "square": -1.0}
LATTICE = {"honeycomb": kite.HONEYCOMB, "square": kite.SQUARE}
ORBITALS = {"honeycomb": 2, "square": 1}
A_CC = 1.0 / math.sqrt(3.0)


def listed():
    return [
        # one small lattice, checked in double precision: the smallest job, where launches count
        dict(name="dos_small_fp64", kind="dos", lattice="honeycomb", Lx=64, Ly=64, W=1.0, gauss=False, delta=0.0,
             p_vac=0.0, M=256, R=4, fp64=True, doubling=False, real=False, flux_steps=0, open_x=False,
             open_y=False, K=1024),
        # an ordinary disorder study: a ragged lattice with vacancies, a few hundred cells a side
        dict(name="dos_vacancies", kind="dos", lattice="honeycomb", Lx=257, Ly=510, W=2.0, gauss=False, delta=0.3,
             p_vac=0.01, M=1024, R=8, fp64=False, doubling=False, real=False, flux_steps=0, open_x=False,
             open_y=False, K=1024),
        # the headline lattice at a quarter of its order
        dict(name="dos_large", kind="dos", lattice="honeycomb", Lx=4096, Ly=4096, W=2.0, gauss=False, delta=0.0,
             p_vac=0.005, M=512, R=8, fp64=False, doubling=False, real=False, flux_steps=0, open_x=False,
             open_y=False, K=1024),
        # double precision on a large lattice, Gaussian disorder, two moments per step
        dict(name="dos_fp64_doubling", kind="dos", lattice="square", Lx=1000, Ly=1001, W=0.3, gauss=True, delta=0.0,
             p_vac=0.0, M=256, R=4, fp64=True, doubling=True, real=False, flux_steps=0, open_x=False,
             open_y=False, K=1024),
        # Landau levels of a strip: a magnetic field and an open edge
        dict(name="landau_strip", kind="dos", lattice="honeycomb", Lx=512, Ly=601, W=0.5, gauss=False, delta=0.0,
             p_vac=0.0, M=512, R=4, fp64=False, doubling=False, real=False, flux_steps=3, open_x=False,
             open_y=True, K=1024),
        # an ensemble of independent square lattices of mixed sizes and orders in one launch
        dict(name="ensemble_square", kind="batch", lattice="square", count=24, sizes=5, L_lo=64, L_hi=1024, M_hi=4096,
             R=4, doubling=False),
        # 2D moments of the conductivity tensor
        dict(name="kubo_moments", kind="kubo", lattice="honeycomb", Lx=512, Ly=512, W=1.0, M=512, R=2, alpha=0, beta=0),
        # optical conductivity from 2D moments
        dict(name="optical_sigma", kind="sigma", M=512, K=128, kT=0.0, jackson=False),
        # Hall conductivity over a window of Fermi energies
        dict(name="hall_dc", kind="hall", M=256, K=48, kT=0.0, jackson=True),
        # ARPES along a path of k-points
        dict(name="arpes_path", kind="arpes", lattice="honeycomb", Lx=300, Ly=300, W=1.0, M=512, nk=24, fp64=False,
             doubling=False),
        # wave packets on a lattice of a million cells
        dict(name="wavepacket", kind="wave", lattice="honeycomb", Lx=1024, Ly=1024, W=1.0, R=4, dt=6.0, nsteps=4,
             fp64=False),
        # densities of many systems from few moments with a trained network
        dict(name="learned_densities", kind="learned", n=1000, mu_ld=512, M_plain=512),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng: random.Random):
    kind = rng.choice(["dos", "dos", "dos", "batch", "kubo", "sigma", "hall", "arpes", "wave", "learned"])
    if kind == "dos":
        lattice = rng.choice(["honeycomb", "square"])
        Lx, Ly = _log(rng, 24, 2048), _log(rng, 24, 2048)
        fp64 = rng.random() < 0.35
        field = rng.random() < 0.25
        real = not field and rng.random() < 0.2
        R = rng.choice([1, 2, 3, 4, 6, 8]) * (2 if real else 1)
        M = _log(rng, 64, 2048)
        cost = Lx * Ly * R * M * (8 if fp64 else 1)
        M = max(64, int(M * min(1.0, 2.0e10 / cost)))
        return dict(kind="dos", lattice=lattice, Lx=Lx, Ly=Ly, W=rng.choice([0.0, 1.0, 2.0]),
                    gauss=rng.random() < 0.2, delta=rng.choice([0.0, 0.3]) if lattice == "honeycomb" else 0.0,
                    p_vac=rng.choice([0.0, 0.0, 0.01]), M=M, R=R, fp64=fp64, doubling=rng.random() < 0.4, real=real,
                    flux_steps=rng.randint(1, 4) if field else 0, open_x=rng.random() < 0.15,
                    open_y=rng.random() < 0.15, K=_log(rng, 100, 4000))
    if kind == "batch":
        return dict(kind="batch", lattice=rng.choice(["honeycomb", "square"]), count=rng.randint(5, 32),
                    sizes=rng.randint(0, 10**6), L_lo=48, L_hi=_log(rng, 128, 700), M_hi=rng.choice([512, 1024, 2048]),
                    R=rng.choice([1, 2, 4, 8]), doubling=rng.random() < 0.4)
    if kind == "kubo":
        return dict(kind="kubo", lattice=rng.choice(["honeycomb", "square"]), Lx=_log(rng, 48, 512),
                    Ly=_log(rng, 48, 512), W=1.0, M=_log(rng, 64, 512), R=rng.randint(1, 2), alpha=rng.randint(0, 1),
                    beta=rng.randint(0, 1))
    if kind == "sigma":
        return dict(kind="sigma", M=_log(rng, 64, 512), K=_log(rng, 20, 128), kT=rng.choice([0.0, 0.05]),
                    jackson=rng.random() < 0.5)
    if kind == "hall":
        return dict(kind="hall", M=_log(rng, 64, 256), K=_log(rng, 5, 48), kT=rng.choice([0.0, 0.02]),
                    jackson=rng.random() < 0.5)
    if kind == "arpes":
        return dict(kind="arpes", lattice=rng.choice(["honeycomb", "square"]), Lx=_log(rng, 40, 300),
                    Ly=_log(rng, 40, 300), W=1.0, M=_log(rng, 64, 512), nk=rng.randint(1, 24), fp64=rng.random() < 0.3,
                    doubling=rng.random() < 0.5)
    if kind == "wave":
        fp64 = rng.random() < 0.4
        return dict(kind="wave", lattice=rng.choice(["honeycomb", "square"]), Lx=_log(rng, 64, 700),
                    Ly=_log(rng, 64, 700), W=1.0, R=rng.choice([1, 2, 3, 4]), dt=rng.choice([1.5, 3.0, 6.0]),
                    nsteps=rng.randint(1, 4), fp64=fp64)
    ld = rng.choice([128, 256, 512])
    return dict(kind="learned", n=_log(rng, 40, 1000), mu_ld=ld, M_plain=rng.choice([128, ld]))


# ---- what a program has in hand ---------------------------------------------------------

_CTX = None


def _context():
    """The one context that a program opens and keeps."""
    global _CTX
    if _CTX is None:
        _CTX = kite.Context(0)
    return _CTX


def _system_seed(seed, i=0):
    return (int(seed) * 1000003 + 7919 * i + 11) & ((1 << 62) - 1)


def _flux(case):
    """A flux that closes on the torus: a whole number of the smallest steps."""
    step = (2.0 if case["lattice"] == "honeycomb" else 1.0) / case["Ly"]
    return case.get("flux_steps", 0) * step


def _system(case, seed):
    return kite.make_system(LATTICE[case["lattice"]], case["Lx"], case["Ly"], t=T_HOP[case["lattice"]], W=case["W"],
                            delta=case.get("delta", 0.0), p_vac=case.get("p_vac", 0.0), seed=_system_seed(seed),
                            disorder=int(case.get("gauss", False)), flux=_flux(case),
                            open_x=int(case.get("open_x", False)), open_y=int(case.get("open_y", False)))


def _members(case, seed):
    """The members of an ensemble: sizes and orders belong to the case, disorder to the seed."""
    g = random.Random(case["sizes"])
    out = []
    for i in range(case["count"]):
        L = g.randint(case["L_lo"], case["L_hi"])
        W = 4.0 * g.random()
        M = g.choice([m for m in (256, 512, 1024, 2048, 4096) if m <= case["M_hi"]])
        out.append(dict(lattice=case["lattice"], Lx=L, Ly=L, W=W, M=M, seed=_system_seed(seed, i)))
    return out


def _toy_moments(M, seed, hall):
    """2D moments of a small random model: states at x_p in (-1, 1) joined by velocity
    matrix elements that fall off with their distance, as those of a disordered metal do."""
    g = np.random.Generator(np.random.PCG64(int(seed) + 17))
    P = 96
    x = np.sort(g.uniform(-0.95, 0.95, P))
    fall = 1.0 / (1.0 + ((x[:, None] - x[None, :]) / 0.2) ** 2)

    def velocity():
        a = g.standard_normal((P, P)) + 1j * g.standard_normal((P, P))
        return 0.5 * (a + a.conj().T) * np.sqrt(fall)

    va = velocity()
    vb = velocity() if hall else va
    C = np.cos(np.arange(M)[:, None] * np.arccos(x)[None, :])
    return np.ascontiguousarray(C @ (va.T * vb) @ C.T / P)


def _k_path(case):
    s = np.linspace(0.0, 1.0, case["nk"])
    return np.ascontiguousarray(np.stack([4.1887902 * s, 1.2 * np.sin(2.0 * s)], axis=1))


def _wave_terms(case):
    lo, hi = _window(case)
    return int(1.1 * 0.5 * (hi - lo) * case["dt"]) + 24


def _packets(case, seed):
    """Gaussian wave packets of random centre and momentum, normalised."""
    g = np.random.Generator(np.random.PCG64(int(seed) + 29))
    s = ORBITALS[case["lattice"]]
    x = torch.arange(case["Lx"], dtype=torch.float64, device=DEV)
    y = torch.arange(case["Ly"], dtype=torch.float64, device=DEV)
    out = []
    for _ in range(case["R"]):
        cx, cy, kx, ky = g.uniform(0.3, 0.7) * case["Lx"], g.uniform(0.3, 0.7) * case["Ly"], *g.uniform(-1, 1, 2)
        sx, sy = 0.12 * case["Lx"], 0.12 * case["Ly"]
        ax = torch.exp(-0.5 * ((x - cx) / sx) ** 2) * torch.exp(1j * kx * x)
        ay = torch.exp(-0.5 * ((y - cy) / sy) ** 2) * torch.exp(1j * ky * y)
        p = (ay[:, None] * ax[None, :])[:, :, None].expand(-1, -1, s)
        out.append((p / torch.linalg.vector_norm(p)).reshape(-1))
    return torch.stack(out).contiguous()


def _network(seed):
    g = np.random.Generator(np.random.PCG64(int(seed) + 41))
    parts = []
    for rows, cols, head in ((512, 128, 1.0), (512, 512, 1.0), (1024, 512, 0.02)):
        lim = math.sqrt(6.0 / cols) * head
        parts += [g.uniform(-lim, lim, rows * cols), g.uniform(-0.01, 0.01, rows)]
    return np.concatenate(parts).astype(np.float32)


def _density_moments(case, seed):
    """Moments of smooth densities with a few peaks; a share of them too sharp for few moments."""
    g = torch.Generator(device=DEV).manual_seed(int(seed) + 53)
    n, P = case["n"], 2048
    th = (torch.arange(P, dtype=torch.float64, device=DEV) + 0.5) * (math.pi / P)
    x = torch.cos(th)
    rho = torch.zeros(n, P, dtype=torch.float64, device=DEV)
    for _ in range(3):
        c = 1.2 * torch.rand(n, 1, generator=g, dtype=torch.float64, device=DEV) - 0.6
        s = 0.25 + 0.2 * torch.rand(n, 1, generator=g, dtype=torch.float64, device=DEV)
        rho += torch.exp(-0.5 * ((x - c) / s) ** 2)
    sharp = torch.rand(n, 1, generator=g, dtype=torch.float64, device=DEV) < 0.02
    rho += sharp * 20.0 * torch.exp(-0.5 * ((x - 0.3) / 0.02) ** 2)
    w = rho * torch.sin(th)
    w = w / w.sum(1, keepdim=True)
    n_ = torch.arange(case["mu_ld"], dtype=torch.float64, device=DEV)
    return (w @ torch.cos(th[:, None] * n_[None, :])).contiguous()


def _norm_stats():
    k = np.arange(128)
    shift = (np.where(k == 0, 1.0, 0.0)).astype(np.float32)
    scale = (1.0 / np.maximum(0.3 / (1.0 + k), 1e-2)).astype(np.float32)
    return shift, scale


LEARNED_WINDOW = (-11.716, 11.716)
SIGMA_WINDOW = (-8.6961, 8.6961)


def prepare(case, seed):
    ctx, kind = _context(), case["kind"]
    s = dict(case=case, ctx=ctx)
    if kind == "dos":
        s["system"] = _system(case, seed)
        s["kpm"] = kite.make_kpm(case["M"], case["R"], 1, kite.FP64 if case["fp64"] else kite.FP32,
                                 doubling=case["doubling"], real_vectors=case["real"])
        s["window"] = kite.bounds(s["system"])
        s["E"] = np.linspace(*s["window"], case["K"] + 2)[1:-1].copy()
    elif kind == "batch":
        m = _members(case, seed)
        s["systems"] = [kite.make_system(LATTICE[c["lattice"]], c["Lx"], c["Ly"], t=T_HOP[c["lattice"]], W=c["W"],
                                         seed=c["seed"]) for c in m]
        s["kpms"] = [kite.make_kpm(c["M"], case["R"], 1, kite.FP32, doubling=case["doubling"]) for c in m]
    elif kind == "kubo":
        s["system"] = _system(case, seed)
        s["kpm"] = kite.make_kpm(case["M"], case["R"], 1, kite.FP32)
    elif kind in ("sigma", "hall"):
        s["mu"] = torch.from_numpy(_toy_moments(case["M"], seed, kind == "hall")).to(DEV)
        s["grid"] = _sigma_grid(case)
    elif kind == "arpes":
        s["system"] = _system(case, seed)
        s["kpm"] = kite.make_kpm(case["M"], 1, 1, kite.FP64 if case["fp64"] else kite.FP32, doubling=case["doubling"])
        s["k"] = _k_path(case)
    elif kind == "wave":
        s["system"] = _system(case, seed)
        s["kpm"] = kite.make_kpm(_wave_terms(case), case["R"], 1, kite.FP64 if case["fp64"] else kite.FP32)
        s["psi0"] = _packets(case, seed)
        s["psi"] = torch.empty_like(s["psi0"])
    else:
        shift, scale = _norm_stats()
        s["model"] = kite.model_import(ctx, _network(seed), *LEARNED_WINDOW, shift=shift, scale=scale)
        s["mu"] = _density_moments(case, seed)
    return s


def _sigma_grid(case):
    hi = SIGMA_WINDOW[1]
    if case["kind"] == "sigma":
        return np.linspace(0.1, 1.4 * hi, case["K"])
    return np.linspace(-0.6 * hi, 0.6 * hi, case["K"])


def run(s):
    case, ctx, kind = s["case"], s["ctx"], s["case"]["kind"]
    if kind == "dos":
        M, K = case["M"], case["K"]
        mu, per = np.zeros(M), np.zeros((case["R"], M, 2))
        kite.moments_1d(ctx, s["system"], s["kpm"], mu, per)
        rho = np.zeros(K)
        kite.reconstruct_dos(ctx, mu, M, M, kite.KERNEL_JACKSON, 0.0, *s["window"], s["E"], K, rho)
        return dict(mu=mu, per_vector=per, rho=rho)
    if kind == "batch":
        mus = [np.zeros(k.M) for k in s["kpms"]]
        kite.moments_1d_batched(ctx, s["systems"], s["kpms"], mus)
        return mus
    if kind == "kubo":
        mu = torch.empty((case["M"], case["M"]), dtype=torch.complex128, device=DEV)
        kite.moments_2d(ctx, s["system"], s["kpm"], mu, case["alpha"], case["beta"])
        return mu
    if kind == "sigma":
        K, M = case["K"], case["M"]
        out = np.zeros(K, dtype=np.complex128)
        kite.reconstruct_sigma(ctx, s["mu"], M, M, kite.HONEYCOMB,
                               kite.KERNEL_JACKSON if case["jackson"] else kite.KERNEL_NONE, *SIGMA_WINDOW, 0.2,
                               case["kT"], 0.1, s["grid"], K, out)
        return out
    if kind == "hall":
        K, M = case["K"], case["M"]
        kern = kite.KERNEL_JACKSON if case["jackson"] else kite.KERNEL_NONE
        hall, dc = np.zeros(K), np.zeros(K)
        kite.reconstruct_sigma_dc_bastin(ctx, s["mu"], M, M, kite.HONEYCOMB, kern, 0.0, *SIGMA_WINDOW, 0.1,
                                         case["kT"], s["grid"], K, hall)
        kite.reconstruct_sigma_dc(ctx, s["mu"], M, M, kite.HONEYCOMB, kern, 0.0, *SIGMA_WINDOW, s["grid"], K, dc)
        return dict(bastin=hall, greenwood=dc)
    if kind == "arpes":
        mu = np.zeros((case["nk"], case["M"], 2))
        kite.spectral_k(ctx, s["system"], s["kpm"], s["k"], case["nk"], mu)
        return mu
    if kind == "wave":
        s["psi"].copy_(s["psi0"])
        norms = np.zeros((case["nsteps"], case["R"]))
        kite.propagate(ctx, s["system"], s["kpm"], case["dt"], case["nsteps"], s["psi"], norms)
        return dict(psi=s["psi"], norms=norms)
    n = case["n"]
    rho = torch.empty((n, kite.MLP_OUT), dtype=torch.float32, device=DEV)
    fell = np.zeros(n, dtype=np.int32)
    dev = np.zeros(n)
    kite.learned_dos(ctx, s["model"], s["mu"], case["mu_ld"], n, 0.05, 16, case["M_plain"], rho, fell, dev)
    return dict(rho=rho, fell_back=fell, deviation=dev)


def work(case):
    """Bytes: the inputs, start vectors and on-site terms that the call itself draws, each once,
    and the outputs.  Flops: the stencil, the moments and the contractions."""
    kind = case["kind"]
    if kind in ("dos", "arpes", "kubo", "wave"):
        N = case["Lx"] * case["Ly"] * ORBITALS[case["lattice"]]
        R = case.get("R", case.get("nk"))
        real = 8 if case.get("fp64") else 4
        lane = 1 if case.get("real") else 2
        # sum of the neighbours, two multiply-adds per real lane
        step = N * R * lane * ((6 if case["lattice"] == "honeycomb" else 7) + (4 if case.get("flux_steps") else 0))
        if kind == "dos":
            steps = case["M"] // 2 if case["doubling"] else case["M"]
            return dict(bytes=N * real * (1 + R * lane) + 8 * (case["M"] * (2 * case["R"] + 1) + 2 * case["K"]),
                        flops=steps * (step + N * R * lane * (4 if case["doubling"] else 2)) + 4 * case["M"] * case["K"])
        if kind == "arpes":
            steps = case["M"] // 2 if case["doubling"] else case["M"]
            return dict(bytes=N * real * (1 + R * lane) + 16 * case["nk"] * case["M"],
                        flops=steps * (step + N * R * lane * (4 if case["doubling"] else 2)))
        if kind == "kubo":
            M = case["M"]
            return dict(bytes=N * real * (1 + 2 * R) + 16 * M * M,
                        flops=R * (8 * M * M * N) + 2 * M * step)
        M = _wave_terms(case)
        return dict(bytes=N * real + 2 * 16 * N * R, flops=case["nsteps"] * M * (step + 4 * N * R))
    if kind == "batch":
        b = f = 0
        for c in _members(case, 0):
            N = c["Lx"] * c["Ly"] * ORBITALS[c["lattice"]]
            b += N * 4 * (1 + 2 * case["R"]) + 8 * c["M"]
            steps = c["M"] // 2 if case["doubling"] else c["M"]
            f += steps * N * case["R"] * 2 * ((6 if c["lattice"] == "honeycomb" else 7) + (4 if case["doubling"] else 2))
        return dict(bytes=b, flops=f)
    if kind == "sigma":
        M, K, Q = case["M"], case["K"], 2 * case["M"] + 64
        return dict(bytes=16 * M * M + 24 * K, flops=2 * 4 * M * M * Q + 2 * K * Q * M * 8)
    if kind == "hall":
        M, K, Q = case["M"], case["K"], 2 * case["M"] + 64
        return dict(bytes=2 * 16 * M * M + 32 * K, flops=K * (4 * M * M * Q + 16 * M * Q) + 2 * M * M * K)
    n = case["n"]
    return dict(bytes=n * (128 * 8 + 4096 + 12) + 4 * 855552, flops=2 * n * (128 * 512 + 512 * 512 + 512 * 1024 + 128 * 1024))


# ---- the same results in 64 bits, from the definitions --------------------------------------

M32 = 0xFFFFFFFF


def _philox(c0, c1, c2, c3, seed):
    """Philox4x32-10 on int64 tensors that hold 32-bit words."""
    k0, k1 = seed & M32, (seed >> 32) & M32
    for r in range(10):
        if r:
            k0, k1 = (k0 + 0x9E3779B9) & M32, (k1 + 0xBB67AE85) & M32
        p0, p1 = c0 * 0xD2511F53, c2 * 0xCD9E8D57  # wraps modulo 2^64: the low 64 bits are right
        c0, c1, c2, c3 = ((p1 >> 32) & M32) ^ c1 ^ k0, p1 & M32, ((p0 >> 32) & M32) ^ c3 ^ k1, p0 & M32
    return c0, c1, c2, c3


def _u53(w0, w1):
    return ((w0 << 21) | (w1 >> 11)).double() * 2.0 ** -53


def _window(case):
    z = 3.0 if case["lattice"] == "honeycomb" else 4.0
    v = (8.58 if case.get("gauss") else 0.5) * case["W"]
    b = (z * abs(T_HOP[case["lattice"]]) + v + 0.5 * abs(case.get("delta", 0.0))) * 1.01
    return -b, b


class _Lattice:
    """H~ of one realisation on [R][Ly][Lx][orbitals] tensors."""

    def __init__(self, case, seed):
        self.c, self.s = case, ORBITALS[case["lattice"]]
        self.Lx, self.Ly, self.seed = case["Lx"], case["Ly"], seed
        self.N = self.Lx * self.Ly * self.s
        lo, hi = _window(case)
        self.plus, self.minus = 0.5 * (hi + lo), 0.5 * (hi - lo)
        self.t = T_HOP[case["lattice"]] / self.minus
        o = torch.arange(self.N, dtype=torch.int64, device=DEV)
        zero = torch.zeros_like(o)
        w = _philox(o, zero, zero, zero + 1, seed)
        if case.get("gauss"):
            v = torch.sqrt(-2.0 * torch.log(1.0 - _u53(w[0], w[1]))) * torch.cos(2.0 * math.pi * w[3].double() * 2.0 ** -32)
            v = case["W"] * v
        else:
            v = case["W"] * (_u53(w[0], w[1]) - 0.5)
        if case.get("delta", 0.0):
            v = v + (0.5 - (o & 1).double()) * case["delta"]
        self.keep = (w[2] >= int(math.floor(case.get("p_vac", 0.0) * 2.0 ** 32)))
        self.n_eff = int(self.keep.sum())
        self.keep = self.keep.reshape(self.Ly, self.Lx, self.s)
        self.v = (((v - self.plus) / self.minus).reshape(self.Ly, self.Lx, self.s)) * self.keep
        self.phase = self._phases() if case.get("flux_steps") else None

    def _phases(self):
        y = torch.arange(self.Ly, dtype=torch.float64, device=DEV)
        f = _flux(self.c)

        def ph(yo, dx, dy, cell):
            th = -2.0 * math.pi * (f / cell) * (yo - 0.5 * dy) * dx
            return torch.polar(torch.ones_like(th), th)[:, None]

        if self.c["lattice"] == "square":
            return ph(y, 1.0, 0.0, 1.0), ph(y, -1.0, 0.0, 1.0)
        cell, h = 0.5 * math.sqrt(3.0), 0.5 * math.sqrt(3.0)
        ya, yb = h * y - 0.5 * A_CC, h * y + 0.5 * A_CC
        return (ph(ya, -0.5, 0.5 * A_CC, cell), ph(ya, 0.5, 0.5 * A_CC, cell), ph(yb, 0.5, -0.5 * A_CC, cell),
                ph(yb, -0.5, -0.5 * A_CC, cell))

    def _move(self, r, dx, dy):
        """r at (x + dx, y + dy), nothing across an open edge."""
        out = torch.roll(r, shifts=(-dy, -dx), dims=(1, 2))
        if dx and self.c.get("open_x"):
            out[:, :, -1 if dx > 0 else 0] = 0
        if dy and self.c.get("open_y"):
            out[:, -1 if dy > 0 else 0] = 0
        return out

    def neighbours(self, r):
        """Per sublattice the neighbours' values with their bond phases."""
        if self.s == 1:
            r = r[..., 0]
            n = [self._move(r, -1, 0), self._move(r, 1, 0), self._move(r, 0, -1), self._move(r, 0, 1)]
            if self.phase:
                n[0], n[1] = n[0] * self.phase[0], n[1] * self.phase[1]
            return [n]
        a, b = r[..., 0], r[..., 1]
        na = [b, self._move(b, 1, -1), self._move(b, 0, -1)]
        nb = [a, self._move(a, -1, 1), self._move(a, 0, 1)]
        if self.phase:
            na[1], na[2] = na[1] * self.phase[0], na[2] * self.phase[1]
            nb[1], nb[2] = nb[1] * self.phase[2], nb[2] * self.phase[3]
        return [na, nb]

    def h(self, r):
        out = torch.empty_like(r)
        for s, n in enumerate(self.neighbours(r)):
            acc = n[0] + n[1]
            for x in n[2:]:
                acc += x
            out[..., s] = acc
            del acc, n
        out *= self.t
        out += self.v * r
        out *= self.keep
        return out

    def velocity(self, r, direction):
        n = self.neighbours(r)
        if self.s == 1:
            d = [[1.0, -1.0, 0.0, 0.0], [0.0, 0.0, 1.0, -1.0]][direction]
            out = sum(w * x for w, x in zip(d, n[0]) if w)[..., None]
        else:
            d = [[0.0, -0.5, 0.5], [-A_CC, 0.5 * A_CC, 0.5 * A_CC]][direction]
            out = torch.stack([sum(w * x for w, x in zip(d, n[0]) if w), -sum(w * x for w, x in zip(d, n[1]) if w)], -1)
        return out * self.t * self.keep

    def random_vectors(self, R, real=False):
        o = torch.arange(self.N, dtype=torch.int64, device=DEV)
        zero = torch.zeros_like(o)
        out = torch.empty((R, self.N), dtype=torch.float64 if real else torch.complex128, device=DEV)
        for v in range(R):
            w = _philox(o, zero, zero + v, zero + 2, self.seed)
            u = _u53(w[0], w[1])
            out[v] = 1.0 - 2.0 * (u >= 0.5).double() if real else torch.polar(torch.ones_like(u), 2.0 * math.pi * u)
        return out.reshape(R, self.Ly, self.Lx, self.s) * self.keep

    def moments(self, r0, M):
        """<r|T_n|r>/N_eff per vector, two per step: T_2n = 2 T_n T_n - T_0."""
        R = r0.shape[0]

        def dot(a, b):
            return torch.stack([torch.linalg.vecdot(a[i].reshape(-1), b[i].reshape(-1)).real for i in range(R)])

        mu = torch.zeros(R, M + 2, dtype=torch.float64, device=DEV)
        prev, cur = r0, self.h(r0)
        mu[:, 0], mu[:, 1] = dot(r0, r0), dot(r0, cur)
        n = 1
        while 2 * n < M:
            nxt = self.h(cur)
            nxt *= 2.0
            nxt -= prev
            mu[:, 2 * n] = 2.0 * dot(cur, cur) - mu[:, 0]
            mu[:, 2 * n + 1] = 2.0 * dot(cur, nxt) - mu[:, 1]
            prev, cur = cur, nxt
            n += 1
        return (mu[:, :M] / self.n_eff).cpu().numpy()


def _jackson(M):
    n, q = np.arange(M), math.pi / (M + 1)
    return ((M - n + 1) * np.cos(q * n) + np.sin(q * n) / math.tan(q)) / (M + 1)


def _density(mu, eps, minus):
    M = mu.shape[-1]
    c = mu * _jackson(M) * np.where(np.arange(M) == 0, 1.0, 2.0)
    T = np.cos(np.arange(M)[:, None] * np.arccos(eps)[None, :])
    return (c @ T) / (math.pi * np.sqrt(1.0 - eps * eps) * minus)


def _exact_sigma(case, seed):
    M, Q = case["M"], 2 * case["M"] + 64
    minus = SIGMA_WINDOW[1]
    mu = torch.from_numpy(_toy_moments(M, seed, case["kind"] == "hall")).to(DEV)
    k = torch.from_numpy(_jackson(M) if case["jackson"] else np.ones(M)).to(DEV)
    half = torch.ones(M, dtype=torch.float64, device=DEV)
    half[0] = 0.5
    A = mu * (k * half)[:, None] * (k * half)[None, :]
    n = torch.arange(M, dtype=torch.float64, device=DEV)
    x, w = (torch.from_numpy(a).to(DEV) for a in np.polynomial.legendre.leggauss(Q))
    ucf, eta, kT = 4.0 / math.sqrt(3.0), 0.1 / minus, case["kT"]

    def nodes(E_F):
        thF = 0.0 if kT else math.acos(E_F / minus)
        th = thF + 0.5 * (math.pi - thF) * (x + 1.0)
        wt = w * 0.5 * (math.pi - thF)
        if kT:
            wt = wt / (1.0 + torch.exp((torch.cos(th) * minus - E_F) / kT))
        return th, (2.0 / math.pi) * torch.cos(n[:, None] * th[None, :]) * wt

    def green(z, sign):
        """CPGF coefficients [M][Q] and sqrt(1 - z^2)."""
        r = torch.sqrt(1.0 - z * z)
        q = z - sign * 1j * r
        return (-2.0j * sign / r)[None, :] * torch.exp(n[:, None] * torch.log(q)[None, :]), r

    out = np.zeros(case["K"], dtype=np.complex128)
    if case["kind"] == "sigma":
        th, D = nodes(0.2)
        G = -A
        U, W = G @ D.to(G.dtype), G.T @ D.to(G.dtype)
        for i, om in enumerate(_sigma_grid(case) / minus):
            gr, _ = green(torch.cos(th) + om + 1j * eta, 1.0)
            ga, _ = green(torch.cos(th) - om - 1j * eta, -1.0)
            out[i] = -1j * ucf / om * complex((gr * U + ga * W).sum())
        return out
    greenwood = np.zeros(case["K"])
    for i, E_F in enumerate(_sigma_grid(case)):
        th, D = nodes(E_F)
        e = torch.cos(th)
        F = 0.0
        for sign, X in ((1.0, A.T), (-1.0, A)):
            z = e + sign * 1j * eta
            g, r = green(z, sign)
            dg = g * (sign * 1j * n[:, None] / r[None, :] + (z / (1.0 - z * z))[None, :])
            F = F + sign * complex((dg * (X @ D.to(X.dtype))).sum())
        out[i] = -ucf * F.imag
        ef = E_F / minus
        c = 2.0 * half * k * torch.cos(n * math.acos(ef)) / (math.pi * math.sqrt(1.0 - ef * ef))
        greenwood[i] = math.pi * ucf * float(c @ mu.real @ c)
    return dict(bastin=out.real.copy(), greenwood=greenwood)


def _exact_wave(case, seed):
    lat, M = _Lattice(case, _system_seed(seed)), _wave_terms(case)
    P = 4 * M
    th = (np.arange(P) + 0.5) * math.pi / P
    f = np.exp(-1j * lat.minus * case["dt"] * np.cos(th))
    c = np.array([(1.0 if n == 0 else 2.0) / P * np.sum(f * np.cos(n * th)) for n in range(M)])
    psi = _packets(case, seed).reshape(case["R"], lat.Ly, lat.Lx, lat.s) * lat.keep
    norms = np.zeros((case["nsteps"], case["R"]))
    for k in range(case["nsteps"]):
        prev, cur = psi, lat.h(psi)
        acc = complex(c[0]) * prev + complex(c[1]) * cur
        for n in range(2, M):
            prev, cur = cur, 2.0 * lat.h(cur) - prev
            acc += complex(c[n]) * cur
        psi = acc
        norms[k] = psi.abs().square().sum((1, 2, 3)).cpu().numpy()
    return dict(psi=psi.reshape(case["R"], -1), norms=norms)


def _exact_learned(case, seed):
    p = torch.from_numpy(_network(seed)).to(DEV).double()
    sizes = [(512, 128), (512, 512), (1024, 512)]
    layers, at = [], 0
    for rows, cols in sizes:
        layers.append((p[at:at + rows * cols].reshape(rows, cols), p[at + rows * cols:at + rows * cols + rows]))
        at += rows * cols + rows
    shift, scale = (torch.from_numpy(a).to(DEV).double() for a in _norm_stats())
    mu = _density_moments(case, seed)
    y = (mu[:, :128] - shift) * scale
    for i, (w, b) in enumerate(layers):
        y = y @ w.T + b
        y = torch.relu(y) if i < 2 else y
    minus = 0.5 * (LEARNED_WINDOW[1] - LEARNED_WINDOW[0])
    eps = -1.0 + (2.0 * np.arange(1024) + 1.0) / 1024
    rho = y.cpu().numpy() + _density(mu[:, :128].cpu().numpy(), eps, minus)
    T = np.cos(np.arange(16)[:, None] * np.arccos(eps)[None, :])
    dev = np.abs(rho * minus @ T.T * (2.0 / 1024) - mu[:, :16].cpu().numpy()).max(1)
    plain = _density(mu[:, :case["M_plain"]].cpu().numpy(), eps, minus)
    return dict(rho=np.where((dev > 0.05)[:, None], plain, rho), fell_back=None, deviation=dev)


def exact(case, seed):
    kind = case["kind"]
    if kind == "dos":
        lat = _Lattice(case, _system_seed(seed))
        re = lat.moments(lat.random_vectors(case["R"], case["real"]), case["M"])
        mu = re.mean(0)
        lo, hi = _window(case)
        eps = np.linspace(lo, hi, case["K"] + 2)[1:-1] / lat.minus
        return dict(mu=mu, per_vector=np.stack([re, np.zeros_like(re)], -1), rho=_density(mu, eps, lat.minus))
    if kind == "batch":
        out = []
        for c in _members(case, seed):
            lat = _Lattice(c, c["seed"])
            out.append(lat.moments(lat.random_vectors(case["R"]), c["M"]).mean(0))
        return out
    if kind == "kubo":
        lat, M = _Lattice(case, _system_seed(seed)), case["M"]
        r = lat.random_vectors(case["R"])
        mu = torch.zeros((M, M), dtype=torch.complex128, device=DEV)
        for v in range(case["R"]):
            fam = []
            for start, after in ((lat.velocity(r[v:v + 1], case["alpha"]), None), (r[v:v + 1], case["beta"])):
                f = torch.empty((M, lat.N), dtype=torch.complex128, device=DEV)
                prev, cur = None, start
                for n in range(M):
                    f[n] = (cur if after is None else lat.velocity(cur, after)).reshape(-1)
                    prev, cur = cur, (lat.h(cur) if n == 0 else 2.0 * lat.h(cur) - prev)
                fam.append(f)
            mu += fam[0].conj() @ fam[1].T
        return mu / (lat.n_eff * case["R"])
    if kind in ("sigma", "hall"):
        return _exact_sigma(case, seed)
    if kind == "arpes":
        lat = _Lattice(case, _system_seed(seed))
        y, x = torch.meshgrid(torch.arange(lat.Ly, dtype=torch.float64, device=DEV),
                              torch.arange(lat.Lx, dtype=torch.float64, device=DEV), indexing="ij")
        if lat.s == 2:
            X = torch.stack([x + 0.5 * y] * 2, -1)
            Y = torch.stack([0.5 * math.sqrt(3.0) * y - 0.5 * A_CC, 0.5 * math.sqrt(3.0) * y + 0.5 * A_CC], -1)
        else:
            X, Y = x[..., None], y[..., None]
        k = _k_path(case)
        r0 = torch.stack([torch.polar(torch.ones_like(X), float(a) * X + float(b) * Y) for a, b in k]) * lat.keep
        re = lat.moments(r0, case["M"])
        return np.stack([re, np.zeros_like(re)], -1)
    if kind == "wave":
        return _exact_wave(case, seed)
    return _exact_learned(case, seed)
