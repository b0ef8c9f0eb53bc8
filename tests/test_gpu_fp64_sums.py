"""The FP64 streaming sweeps: one, two or three steps a pass, complex and real start vectors,
every chunk count, plain moments and moment doubling, each vector's moments against the
oracle.  Both sides run the recursion in FP64 (40 steps, |r_n| <= |r_0| per state: rounding
of 40 * 4 * 2^-53 of the norm, 2e-14) and sum at most 66 000 terms of a sum of absolute
values <= 1 (2^-53 per addition along chains of at most 400): 1e-12 covers both."""
import contextlib
import os

import numpy as np
import pytest

import oracle

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


# a strip of a single cell column at the right edge, rows past 32 and fewer rows than CTAs
SIZES = [(kite.HONEYCOMB, 129, 37), (kite.HONEYCOMB, 33, 1000), (kite.SQUARE, 257, 41), (kite.SQUARE, 65, 1000)]


@pytest.mark.parametrize("lat,Lx,Ly", SIZES)
@pytest.mark.parametrize("steps,doubling", [("1", False), ("2", False), ("3", False), ("1", True), ("2", True)])
@pytest.mark.parametrize("R,real", [(1, False), (2, False), (3, False), (2, True), (8, True)])
def test_every_vector_against_the_oracle(ctx, lat, Lx, Ly, steps, doubling, R, real):
    d = dict(lattice=lat, Lx=Lx, Ly=Ly, t=-2.7 if lat == kite.HONEYCOMB else -1.0, W=1.5, p_vac=0.02, seed=5)
    M = 41
    o = oracle.make_system(**d)
    ref = oracle.moments_1d(o, M, R, r0=oracle.random_real(o, R) if real else None)
    mu, muv = np.zeros(M), np.zeros((R, M, 2))
    with env(KITE_RESIDENT="0", KITE_CLUSTER="0", KITE_PASS_STEPS=steps):
        st = kite.moments_1d(ctx, kite.make_system(**d),
                             kite.make_kpm(M, R, 1, kite.FP64, doubling=doubling, real_vectors=real), mu, muv)
    assert st.cluster_ctas == 0
    assert np.max(np.abs(muv[..., 0] - ref.real)) <= 1e-12
    assert np.all(muv[..., 1] == 0.0)
    assert np.max(np.abs(mu - ref.real.mean(0))) <= 1e-12
