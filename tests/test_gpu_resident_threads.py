"""On-chip sweeps of several contexts at once, each with its own stream and host thread, beside
batched sweeps and time evolutions: a sweep takes every SM and its CTAs wait on one another, so
it must not start in part.  Every call succeeds and repeats its own bits."""
import threading

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

kite = pytest.importorskip("paper_1910_05194_gb300")


def sweep(i, out):
    d = dict(lattice=i % 2, Lx=180 + 10 * i, Ly=150, t=-1.0, W=1.0, seed=i + 1)
    k = kite.make_kpm(96, 4, 1, (i // 2) % 2)
    with kite.Context(0) as ctx:
        for _ in range(40):
            per = np.zeros((4, 96, 2))
            st = kite.moments_1d(ctx, kite.make_system(**d), k, np.zeros(96), per)
            out.append((per, st.block))


def batch(i, out):
    s = [kite.make_system(kite.SQUARE, 64 + 8 * j, 64, t=-1.0, W=1.0, seed=j + 1) for j in range(6)]
    with kite.Context(0) as ctx:
        for _ in range(20):
            mus = [np.zeros(64) for _ in s]
            kite.moments_1d_batched(ctx, s, [kite.make_kpm(64, 2, 1, kite.FP32)] * 6, mus)
            out.append((np.concatenate(mus), 0))


def evolve(i, out):
    psi0 = np.random.default_rng(1).standard_normal((1, 300 * 200, 2)) / 250
    with kite.Context(0) as ctx:
        for _ in range(20):
            psi = psi0.copy()
            kite.propagate(ctx, kite.make_system(kite.SQUARE, 300, 200, t=-1.0, W=1.0, seed=9),
                           kite.make_kpm(30, 1, 1, kite.FP32), 0.3, 2, psi)
            out.append((psi, 0))


def test_contexts_side_by_side(monkeypatch):
    monkeypatch.setenv("KITE_RESIDENT", "1")
    work = [sweep, sweep, sweep, sweep, batch, evolve]
    outs, errors = [[] for _ in work], []

    def run(f, i):
        try:
            f(i, outs[i])
        except Exception as e:  # noqa: BLE001
            errors.append(e)

    threads = [threading.Thread(target=run, args=(f, i)) for i, f in enumerate(work)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
    for f, out in zip(work, outs):
        assert all(np.array_equal(v, out[0][0]) for v, _ in out)
        if f is sweep:
            assert all(b > 256 for _, b in out)  # none fell back to the streaming kernels
