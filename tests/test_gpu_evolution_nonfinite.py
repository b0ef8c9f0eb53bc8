"""Time evolution of states that are not finite: the pass of two steps leaves the values that
single steps leave (vacancies stay zero), and in FP64, where the series skips the parts of its
coefficients that are zero, a component that is not finite still spoils both parts of its site
(zero times it is NaN)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

kite = pytest.importorskip("paper_1910_05194_gb300")


def evolve(d, M, precision, value, where, part):
    n = d["Lx"] * d["Ly"] * (2 if d["lattice"] == kite.HONEYCOMB else 1)
    psi = np.random.default_rng(5).standard_normal((3, n, 2)) / np.sqrt(n)
    psi[1, where, part] = value
    with kite.Context(0) as ctx:
        kite.propagate(ctx, kite.make_system(**d), kite.make_kpm(M, 3, 1, precision), 0.4, 1, psi)
    return psi


@pytest.mark.parametrize("value", [np.nan, np.inf])
@pytest.mark.parametrize("lattice", [kite.HONEYCOMB, kite.SQUARE])
@pytest.mark.parametrize("M", [4, 7, 12])
def test_passes_and_single_steps_agree(monkeypatch, lattice, value, M):
    d = dict(lattice=lattice, Lx=61, Ly=40, t=-1.0, W=1.0, p_vac=0.3, seed=3)
    a = evolve(d, M, kite.FP32, value, 777, 0)
    monkeypatch.setenv("KITE_PASS_STEPS", "1")
    b = evolve(d, M, kite.FP32, value, 777, 0)
    assert not np.isfinite(a[1]).all() and np.isfinite(a[[0, 2]]).all()
    assert np.array_equal(np.isfinite(a), np.isfinite(b)) and np.array_equal(a[np.isfinite(a)], b[np.isfinite(b)])


@pytest.mark.parametrize("part", [0, 1])
@pytest.mark.parametrize("lattice", [kite.HONEYCOMB, kite.SQUARE])
@pytest.mark.parametrize("M", [2, 3, 9])
def test_fp64_spoils_both_parts(lattice, part, M):
    d = dict(lattice=lattice, Lx=30, Ly=24, t=-1.0, W=1.0, seed=3)
    for value in (np.nan, np.inf):
        bad = ~np.isfinite(evolve(d, M, kite.FP64, value, 300, part))
        assert bad[1].any() and np.array_equal(bad[1, :, 0], bad[1, :, 1]) and not bad[[0, 2]].any()
