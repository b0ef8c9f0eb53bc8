"""What a call does when the on-chip sweep of a mid-size lattice cannot run: the streaming
kernels take over, the moments are those of a call that never tried (the same tuned shape: the
same bits), and nothing is decided from a failed timing.  The failures are made by the hook
kite_debug_fail_resident: a launch reported as refused, or a bounded wait that runs out and
returns a status."""
import contextlib
import os

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

kite = pytest.importorskip("paper_1910_05194_gb300")

LATTICES = [dict(lattice=kite.HONEYCOMB, Lx=200, Ly=220, t=-2.7, W=1.0, seed=5),
            dict(lattice=kite.SQUARE, Lx=200, Ly=201, t=-1.0, W=1.0, seed=5, flux=2.0 / 201)]


@contextlib.contextmanager
def env(**kw):
    old = {k: os.environ.get(k) for k in kw}
    os.environ.update(kw)
    try:
        yield
    finally:
        for k, v in old.items():
            os.environ.pop(k, None) if v is None else os.environ.__setitem__(k, v)


def call(ctx, d, precision, R=4, M=64):
    mu, per = np.zeros(M), np.zeros((R, M, 2))
    st = kite.moments_1d(ctx, kite.make_system(**d), kite.make_kpm(M, R, 1, precision), mu, per)
    return per, st.block


@contextlib.contextmanager
def fresh(d, precision, R=4):
    """A context of its own, with the streaming sweep's moments and the two paths' block sizes."""
    with kite.Context(0) as ctx:
        with env(KITE_RESIDENT="0"):
            ref, stream = call(ctx, d, precision, R)
        with env(KITE_RESIDENT="1"):
            chip = call(ctx, d, precision, R)[1]
        assert stream == 256 < chip  # how kite_stats tells them apart
        yield ctx, ref, stream, chip


@pytest.mark.parametrize("precision", [kite.FP32, kite.FP64])
@pytest.mark.parametrize("d", LATTICES)
@pytest.mark.parametrize("count", [1, 100])
def test_a_failed_timing_decides_nothing(d, precision, count):
    with fresh(d, precision) as (ctx, ref, stream, chip):
        kite.debug_fail_resident(ctx, kite.FAIL_LAUNCH, 0, count)
        per, block = call(ctx, d, precision)
        assert block == stream and np.array_equal(per, ref)
        kite.debug_fail_resident(ctx, kite.FAIL_LAUNCH, 0, 0)
        assert call(ctx, d, precision)[1] == chip  # timed again: faster at these sizes


@pytest.mark.parametrize("precision", [kite.FP32, kite.FP64])
@pytest.mark.parametrize("d", LATTICES)
@pytest.mark.parametrize("skip,count", [(0, 1), (2, 1), (0, 2), (2, 2)])
def test_a_wait_that_runs_out_in_a_timing_run_does_not_fail_the_call(d, precision, skip, count):
    with fresh(d, precision) as (ctx, ref, stream, chip):
        kite.debug_fail_resident(ctx, kite.FAIL_WAIT, skip, count)
        per, block = call(ctx, d, precision)
        assert block == stream and np.array_equal(per, ref)
        kite.debug_fail_resident(ctx, kite.FAIL_WAIT, 0, 0)
        assert call(ctx, d, precision)[1] == chip


@pytest.mark.parametrize("kind", [kite.FAIL_LAUNCH, kite.FAIL_WAIT])
@pytest.mark.parametrize("precision", [kite.FP32, kite.FP64])
@pytest.mark.parametrize("d", LATTICES)
@pytest.mark.parametrize("pinned", [False, True])
def test_a_failed_sweep_goes_to_the_streaming_kernels(d, precision, kind, pinned):
    with fresh(d, precision, 16) as (ctx, ref, stream, chip):  # two or four batches
        assert call(ctx, d, precision, 16)[1] == chip
        with env(**({"KITE_RESIDENT": "1"} if pinned else {})):
            kite.debug_fail_resident(ctx, kind, 0, 1)
            per, block = call(ctx, d, precision, 16)
            assert block == stream and np.array_equal(per, ref)
            assert kite.lib().kite_last_error(ctx.handle) == b""
            assert call(ctx, d, precision, 16)[1] == chip


@pytest.mark.parametrize("d", LATTICES)
def test_a_sweep_that_keeps_failing_is_tried_once_a_call_and_three_times_in_all(d):
    with fresh(d, kite.FP32, 16) as (ctx, ref, stream, chip):
        assert call(ctx, d, kite.FP32, 16)[1] == chip
        for n, left in ((2, "one is left after the first batch"), (1, "the third failure")):
            kite.debug_fail_resident(ctx, kite.FAIL_WAIT, 0, n)
            for _ in range(n):
                per, block = call(ctx, d, kite.FP32, 16)
                assert block == stream and np.array_equal(per, ref), left
        per, block = call(ctx, d, kite.FP32, 16)
        assert block == stream and np.array_equal(per, ref)


@pytest.mark.parametrize("M", [4, 8])
def test_a_short_sweep_is_not_taken_on_chip_where_its_launch_costs_more(M):
    """64 x 64 honeycomb cells, FP64, R = 4: on chip a step gains 0.4 us on the cluster sweep's 2.3,
    a sweep's launch and host part cost 14 us more: some 30 steps bring them in, three and seven
    do not, before and after a longer call of the size."""
    d = dict(lattice=kite.HONEYCOMB, Lx=64, Ly=64, t=-2.7, W=1.0, seed=5)
    with kite.Context(0) as ctx:
        for _ in range(2):
            assert call(ctx, d, kite.FP64, 4, M)[1] == 256
            call(ctx, d, kite.FP64, 4, 300)


@pytest.mark.parametrize("kind,skip,count", [(0, 0, 1), (3, 0, 1), (1, -1, 1), (2, 0, -1)])
def test_the_hook_refuses_what_it_does_not_know(kind, skip, count):
    with kite.Context(0) as ctx, pytest.raises(kite.KiteError) as e:
        kite.debug_fail_resident(ctx, kind, skip, count)
    assert e.value.status == kite.ERR_ARG
