"""The on-chip sweep on both sides of the edge-list length (512 entries a region) at which its exchange
threads take three sites each instead of two: lattices of growing width, whose regions' lists grow
through it for every number of vectors.  The last iterates are the streaming sweep's bits."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

kite = pytest.importorskip("paper_1910_05194_gb300")


def last(monkeypatch, lattice, Lx, R, precision, resident):
    monkeypatch.setenv("KITE_RESIDENT", resident)
    monkeypatch.setenv("KITE_CLUSTER", "0")
    M, Ly = 9, 210
    n = Lx * Ly * (2 if lattice == kite.HONEYCOMB else 1)
    out = np.zeros((R, 2, n), np.complex64 if precision == kite.FP32 else np.complex128)
    s = kite.make_system(lattice, Lx, Ly, t=-1.0, W=1.0, p_vac=0.01, seed=Lx)
    with kite.Context(0) as ctx:
        st = kite.moments_1d(ctx, s, kite.make_kpm(M, R, 1, precision, r_last=out), np.zeros(M))
    return out, st.block


@pytest.mark.parametrize("precision,lattice,widths,R", [
    (kite.FP32, kite.HONEYCOMB, range(90, 400, 31), 8), (kite.FP32, kite.HONEYCOMB, range(150, 640, 61), 4),
    (kite.FP32, kite.SQUARE, range(130, 900, 97), 8), (kite.FP64, kite.HONEYCOMB, range(40, 300, 29), 4),
    (kite.FP64, kite.SQUARE, range(60, 500, 61), 2)])
def test_edge_lists_of_every_length(monkeypatch, precision, lattice, widths, R):
    chip = 0
    for Lx in widths:
        a, block = last(monkeypatch, lattice, Lx, R, precision, "1")
        b, stream = last(monkeypatch, lattice, Lx, R, precision, "0")
        assert stream == 256 and np.array_equal(a.view(np.uint8), b.view(np.uint8))
        chip += block > 256
    assert chip >= len(widths) - 2  # (the widest may not fit)
