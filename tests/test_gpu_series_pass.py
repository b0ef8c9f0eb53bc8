"""FP32 time evolution with two recursion steps per pass and the series added every second
pass: the same additions in the same order as one step per launch (KITE_PASS_STEPS=1), so the
wave functions are the same bits; every remainder of the schedule (M - 2 steps after the first,
in fours, twos and ones), narrow and ragged lattices, every batch shape, vacancies.  FP64 with a
window that is not symmetric (complex coefficients) against the oracle at test_gpu_propagate.py's
1e-10."""
import os

import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu

kite = pytest.importorskip("paper_1910_05194_gb300")


@pytest.fixture(scope="module")
def ctx():
    c = kite.Context(0)
    yield c
    c.close()


def evolve(ctx, d, M, R, nsteps, precision=0, window=(0.0, 0.0), pin=None):
    n = d["Lx"] * d["Ly"] * (2 if d["lattice"] == kite.HONEYCOMB else 1)
    psi0 = synth.gaussian_vectors(n, R, seed=n + R) / np.sqrt(n)
    psi = np.ascontiguousarray(np.stack([psi0.real, psi0.imag], -1))
    norms = np.zeros((nsteps, R))
    if pin:
        os.environ["KITE_PASS_STEPS"] = pin
    try:
        kite.propagate(ctx, kite.make_system(**d), kite.make_kpm(M, R, 1, precision, *window), 0.8, nsteps, psi, norms)
    finally:
        os.environ.pop("KITE_PASS_STEPS", None)
    return psi0, psi, norms


CASES = [(0, 37, 29, 3, 0.02), (0, 130, 65, 1, 0.0), (0, 64, 300, 9, 0.0), (1, 41, 33, 4, 0.05), (1, 300, 17, 8, 0.0),
         (0, 1, 12, 2, 0.0), (1, 3, 3, 1, 0.0), (0, 33, 1, 2, 0.0)]


@pytest.mark.parametrize("M", [3, 4, 5, 6, 7, 8, 9, 24])
@pytest.mark.parametrize("case", CASES)
def test_passes_give_the_bits_of_single_steps(ctx, case, M):
    lat, Lx, Ly, R, p = case
    d = dict(lattice=lat, Lx=Lx, Ly=Ly, t=-1.0, W=1.0, p_vac=p, seed=3)
    a, b = evolve(ctx, d, M, R, 2), evolve(ctx, d, M, R, 2, pin="1")
    assert np.array_equal(a[1], b[1]) and np.array_equal(a[2], b[2])


def test_fp64_series_with_complex_coefficients(ctx):
    for lat in (0, 1):
        d = dict(lattice=lat, Lx=14, Ly=11, t=-1.0, W=1.0, p_vac=0.02, seed=5)
        for window in ((0.0, 0.0), (-4.9, 6.1)):
            psi0, psi, norms = evolve(ctx, d, 40, 2, 2, kite.FP64, window)
            s = oracle.make_system(**d)
            _, vac = oracle.disorder(s)
            lo, hi = window if window[1] else (None, None)
            for v in range(2):
                ref = oracle.propagate(s, psi0[v] * (vac == 0), 0.8, 2, 40, e_min=lo, e_max=hi)[-1]
                assert np.max(np.abs(psi[v, :, 0] + 1j * psi[v, :, 1] - ref)) <= 1e-10
