"""The environment switches of the FP32 time evolution: KITE_AUTOTUNE=0 and KITE_PASS_STEPS=1
take one recursion step per launch, KITE_PASS_STEPS=2 and no switch at all two per pass after the
first; the wave functions are the same bits."""
import os

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

kite = pytest.importorskip("paper_1910_05194_gb300")


def evolve(monkeypatch, M, nsteps, **env):
    for k in ("KITE_AUTOTUNE", "KITE_PASS_STEPS"):
        monkeypatch.delenv(k, raising=False)
    for k, v in env.items():
        monkeypatch.setenv(k, v)
    Lx, Ly = 41, 33
    psi = np.random.default_rng(3).standard_normal((2, 2 * Lx * Ly, 2)) / Lx
    s = kite.make_system(kite.HONEYCOMB, Lx, Ly, t=-2.7, W=1.0, seed=2)
    with kite.Context(0) as ctx:
        st = kite.propagate(ctx, s, kite.make_kpm(M, 2, 1, kite.FP32), 0.2, nsteps, psi)
    return psi, st.step_launches


def test_switches_of_the_time_evolution(monkeypatch):
    M, n = 30, 2
    single, passes = n * (M - 1), n * (1 + (M - 2) // 2)
    ref, launches = evolve(monkeypatch, M, n)
    assert launches == passes
    for env, want in ((dict(KITE_AUTOTUNE="0"), single), (dict(KITE_PASS_STEPS="1"), single),
                      (dict(KITE_PASS_STEPS="2"), passes), (dict(KITE_AUTOTUNE="0", KITE_PASS_STEPS="2"), passes),
                      (dict(KITE_AUTOTUNE="1"), passes)):
        psi, launches = evolve(monkeypatch, M, n, **env)
        assert launches == want and np.array_equal(psi, ref), env
