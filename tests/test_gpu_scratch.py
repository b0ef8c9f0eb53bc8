"""Calls whose work space is limited (a hook refuses more, as a device without room does): where the
faster path's does not fit, the path that needs less runs, with the same results, and the call is
refused only when that one does not fit either."""
import contextlib
import os

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
kite = pytest.importorskip("paper_1910_05194_gb300")

MiB = 1 << 20


@contextlib.contextmanager
def env(**kw):
    old = {k: os.environ.get(k) for k in kw}
    os.environ.update(kw)
    try:
        yield
    finally:
        for k, v in old.items():
            os.environ.pop(k, None) if v is None else os.environ.__setitem__(k, v)


def moments(ctx, M, R=8):
    s = kite.make_system(kite.HONEYCOMB, 257, 510, t=-2.7, W=2.0, seed=3)
    mu, per = np.zeros(M), np.zeros((R, M, 2))
    st = kite.moments_1d(ctx, s, kite.make_kpm(M, R, 1, kite.FP32), mu, per)
    return per, st.block


def test_moments_without_room_for_the_on_chip_sweeps_partials():
    """262140 orbitals, eight vectors, M = 8192: five vector buffers of 17 MB and partials of 152
    CTAs times the streaming grid's CTAs per SM (3 to 5), 16 sums and 8 bytes a step: 0.5 to
    0.9 GB; on chip 152 x 8 instead: 1.3 GB and 0.03 GB of records."""
    M = 8192
    with kite.Context(0) as ctx:
        with env(KITE_RESIDENT="0"):
            ref, stream = moments(ctx, M)
        short = moments(ctx, 64)[1]
    assert short != stream  # on chip where there is room
    with kite.Context(0) as ctx:
        with env(KITE_RESIDENT="0"):
            moments(ctx, 64)  # the same tuned shape
        kite.debug_limit_workspace(ctx, 1240 * MiB)
        per, block = moments(ctx, M)
        assert kite.lib().kite_last_error(ctx.handle) == b""
        assert block == stream and np.max(np.abs(per - ref)) <= 1e-6
        kite.debug_limit_workspace(ctx, 64 * MiB)
        with pytest.raises(kite.KiteError) as e:
            moments(ctx, M)
        assert e.value.status == kite.ERR_OOM
        kite.debug_limit_workspace(ctx, 0)
        assert moments(ctx, M)[1] == short


def test_time_evolution_without_room_for_two_steps_a_pass():
    """3.2 million cells, eight packets: a vector buffer has 205 MB; single steps take four of
    them and 13 MB (0.83 GB), two steps a pass two more (1.24 GB).  The bits are the same."""
    L, R, M = 1789, 8, 12
    s = kite.make_system(kite.SQUARE, L, L, t=-1.0, W=1.0, seed=4)
    g = torch.Generator(device="cuda").manual_seed(1)
    psi0 = torch.randn(R, L * L, 2, dtype=torch.float64, device="cuda", generator=g) / L
    ref, psi = psi0.clone(), psi0.clone()
    norms = np.zeros((2, 1, R))
    with kite.Context(0) as ctx:
        kite.propagate(ctx, s, kite.make_kpm(M, R, 1, kite.FP32), 0.4, 1, ref, norms[0])
    with kite.Context(0) as ctx:
        kite.debug_limit_workspace(ctx, 1050 * MiB)
        st = kite.propagate(ctx, s, kite.make_kpm(M, R, 1, kite.FP32), 0.4, 1, psi, norms[1])
        assert st.step_launches == M - 1 and kite.lib().kite_last_error(ctx.handle) == b""
    assert torch.equal(ref, psi) and np.array_equal(norms[0], norms[1])
    with kite.Context(0) as ctx:
        kite.debug_limit_workspace(ctx, 700 * MiB)
        with pytest.raises(kite.KiteError) as e:
            kite.propagate(ctx, s, kite.make_kpm(M, R, 1, kite.FP32), 0.4, 1, psi)
        assert e.value.status == kite.ERR_OOM
