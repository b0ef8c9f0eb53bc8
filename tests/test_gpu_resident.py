"""The sweep held on chip by the whole GPU, a region of the lattice per SM: KITE_RESIDENT=1
forces it where the lattice fits, KITE_RESIDENT=0 keeps the streaming kernels.  Both apply
the same rounding sequence per site, so the iterates are the same bits.  The moments differ
from an untuned streaming launch by the regrouping of their partial sums only (FP32 over at
most 32 rows on either path, a chain of 64 products: 64 * 2^-24 of sum |terms| / N_eff <= 1
at worst, in the mean far below; the bar between two FP32 paths is 1e-6, FP64 1e-12), and
from the streaming launch of the tuned shape, whose grouping they keep, by the rounding of
FP64 sums (2^-53 of sum |terms| / N_eff <= 1 per addition: far inside 1e-12)."""
import contextlib
import os

import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu

kite = pytest.importorskip("paper_1910_05194_gb300")


@pytest.fixture(scope="module")
def ctx():
    c = kite.Context(0)
    yield c
    c.close()


@contextlib.contextmanager
def env(**kw):
    old = {k: os.environ.get(k) for k in kw}
    os.environ.update(kw)
    try:
        yield
    finally:
        for k, v in old.items():
            os.environ.pop(k, None) if v is None else os.environ.__setitem__(k, v)


def start(d, n, R):
    r0 = synth.gaussian_vectors(n, R, seed=d["Lx"] + 7 * d["Ly"])
    r0 = np.ascontiguousarray(np.stack([r0.real, r0.imag], -1))
    # mu_0 has to stay below 1 over the non-vacant orbitals alone
    r0 *= 0.9 / np.sqrt((r0 ** 2).sum((1, 2), keepdims=True) / n)
    return r0


def run(ctx, d, M, R, resident, precision, want_last=False, **kw):
    s = kite.make_system(**d)
    n = d["Lx"] * d["Ly"] * (2 if d["lattice"] == kite.HONEYCOMB else 1)
    last = np.zeros((R, 2, n), np.complex64 if precision == kite.FP32 else np.complex128) if want_last else None
    r0 = start(d, n, R)
    mu, muv = np.zeros(M), np.zeros((R, M, 2))
    extra = {} if resident else {"KITE_CLUSTER": "0", "KITE_AUTOTUNE": "0"}
    with env(KITE_RESIDENT="1" if resident else "0", **extra):
        st = kite.moments_1d(ctx, s, kite.make_kpm(M, R, 1, precision, r0=r0, r_last=last, **kw), mu, muv)
    return mu, muv, last, st


def launch(r):
    return r[3].grid, r[3].block


def sysd(lat, Lx, Ly, **kw):
    return dict(dict(lattice=lat, Lx=Lx, Ly=Ly, t=-2.7 if lat == kite.HONEYCOMB else -1.0, W=2.0, seed=7), **kw)


HC, SQ = kite.HONEYCOMB, kite.SQUARE
# ragged regions, regions of a few cells, long thin lattices, r_0 read from L2, open
# boundaries, a field, vacancies, every chunk count and a batch in several sweeps
CASES = [
    (sysd(HC, 37, 29, p_vac=0.03), 3, 24), (sysd(SQ, 37, 29), 8, 25), (sysd(HC, 8, 300), 1, 20),
    (sysd(SQ, 301, 9, p_vac=0.05), 2, 20), (sysd(HC, 9, 8), 5, 16), (sysd(SQ, 20, 20), 1, 5),
    (sysd(HC, 257, 255, p_vac=0.01), 8, 14), (sysd(HC, 400, 380), 4, 10), (sysd(SQ, 500, 501), 9, 9),
    (sysd(HC, 64, 64, open_x=1), 4, 20), (sysd(HC, 65, 40, open_y=1, p_vac=0.02), 2, 20),
    (sysd(SQ, 40, 33, open_x=1, open_y=1), 3, 20), (sysd(HC, 48, 60, flux=2.0 / 60), 3, 20),
    (sysd(SQ, 50, 60, flux=3.0 / 60, open_x=1), 4, 20), (sysd(HC, 90, 61, flux=0.013, open_y=1), 1, 20),
    # three edge sites per exchange thread; half chunks (FP32: too large for whole ones)
    (sysd(SQ, 701, 640), 3, 7), (sysd(SQ, 1000, 903, p_vac=0.01), 5, 6), (sysd(HC, 620, 900, open_x=1), 2, 6),
]


@pytest.mark.parametrize("precision", [kite.FP32, kite.FP64])
@pytest.mark.parametrize("case", CASES)
def test_resident_sweep_has_the_streaming_bits(ctx, case, precision):
    d, R, M = case
    if precision == kite.FP64 and d["Lx"] * d["Ly"] > 500_000:
        pytest.skip("does not fit in double precision")
    a = run(ctx, d, M, R, True, precision, want_last=True)
    b = run(ctx, d, M, R, False, precision, want_last=True)
    assert launch(a) != launch(b)
    u = np.uint32 if precision == kite.FP32 else np.uint64
    assert np.array_equal(a[2].view(u), b[2].view(u))
    tol = 1e-6 if precision == kite.FP32 else 1e-12
    assert np.max(np.abs(a[1][..., 0] - b[1][..., 0])) <= tol and np.max(np.abs(a[0] - b[0])) <= tol
    assert a[3].n_eff == b[3].n_eff


@pytest.mark.parametrize("precision", [kite.FP32, kite.FP64])
@pytest.mark.parametrize("kw", [dict(doubling=True), dict(real_vectors=True), dict(doubling=True, real_vectors=True)])
def test_resident_doubling_and_real_vectors(ctx, kw, precision):
    tol = 2e-6 if precision == kite.FP32 else 1e-12  # 2 slot - mu: twice the bar
    for d, R, M in ((sysd(HC, 70, 55, p_vac=0.02), 5, 31), (sysd(SQ, 90, 41, open_y=1), 8, 32)):
        a, b = run(ctx, d, M, R, True, precision, **kw), run(ctx, d, M, R, False, precision, **kw)
        assert launch(a) != launch(b) and np.max(np.abs(a[1][..., 0] - b[1][..., 0])) <= tol


@pytest.mark.parametrize("d,R,M,kw", [
    (sysd(HC, 257, 510, p_vac=0.01), 8, 24, {}), (sysd(HC, 300, 300), 7, 20, dict(doubling=True)),
    (sysd(SQ, 500, 301, p_vac=0.02), 4, 20, {}), (sysd(HC, 200, 220, flux=2.0 / 220), 3, 20, {}),
    (sysd(SQ, 260, 400), 16, 20, dict(real_vectors=True)), (sysd(SQ, 200, 700), 1, 20, dict(doubling=True)),
    (sysd(SQ, 1001, 900), 3, 10, {}), (sysd(HC, 700, 801), 8, 10, dict(doubling=True)),
    (sysd(SQ, 1000, 950), 6, 10, dict(real_vectors=True)), (sysd(SQ, 900, 900, flux=2.0 / 900), 3, 10, {})])
def test_resident_fp32_moments_keep_the_streaming_grouping(d, R, M, kw):
    with kite.Context(0) as c, env(KITE_CLUSTER="0"):  # one context: one tuned shape
        a = run(c, d, M, R, True, kite.FP32, **kw)
        with env(KITE_RESIDENT="0"):
            mu, muv = np.zeros(M), np.zeros((R, M, 2))
            n = d["Lx"] * d["Ly"] * (2 if d["lattice"] == HC else 1)
            r0 = start(d, n, R)  # (the call keeps the address only)
            kite.moments_1d(c, kite.make_system(**d), kite.make_kpm(M, R, 1, kite.FP32, r0=r0, **kw), mu, muv)
    assert np.max(np.abs(a[1] - muv)) <= 1e-12


def test_resident_sweep_is_deterministic_and_follows_a_changed_input(ctx):
    d = sysd(HC, 130, 77)
    a, b = run(ctx, d, 40, 4, True, kite.FP32), run(ctx, d, 40, 4, True, kite.FP32)
    c = run(ctx, dict(d, seed=8), 40, 4, True, kite.FP32)
    assert np.array_equal(a[1], b[1]) and not np.array_equal(a[1], c[1])


def test_resident_bounded_wait_reports_and_leaves_the_context_usable(ctx):
    d = sysd(HC, 64, 64)
    ref = run(ctx, d, 20, 2, True, kite.FP32)
    kite.debug_stall_once(ctx)
    with pytest.raises(kite.KiteError) as e:
        run(ctx, d, 20, 2, True, kite.FP32)
    assert e.value.status == kite.ERR_TIMEOUT
    assert np.array_equal(run(ctx, d, 20, 2, True, kite.FP32)[1], ref[1])
