"""The learned path's Chebyshev sums over many rows (the residual prior and the plain
fallback, one kernel with eight rows per block from 512 rows on and one row below) at the
edges of their tiles: odd and smallest orders, orders across the 128-moment tile, row counts
around 512 and off a multiple of eight, the order above which the fallback goes row by row.
Bar: FP32 outputs of FP64 sums, half a unit in the last place each (2^-24 of the value), plus
the FP64 sums' own rounding of at most M 2^-53 sum |c T|, far below: 2e-7 of the row's largest
value."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

kite = pytest.importorskip("paper_1910_05194_gb300")
LO, HI = -11.0, 12.5
EPS = -1.0 + (2.0 * np.arange(1024) + 1.0) / 1024


@pytest.fixture(scope="module")
def ctx():
    c = kite.Context(0)
    yield c
    c.close()


def jackson_density(mu):
    M = mu.shape[1]
    n, q = np.arange(M), np.pi / (M + 1)
    g = ((M - n + 1) * np.cos(q * n) + np.sin(q * n) / np.tan(q)) / (M + 1) * np.where(n == 0, 1.0, 2.0)
    T = np.cos(n[:, None] * np.arccos(EPS)[None, :])
    return (mu * g) @ T / (np.pi * np.sqrt(1.0 - EPS ** 2) * 0.5 * (HI - LO))


def moments(n, M, seed):
    g = np.random.Generator(np.random.PCG64(seed))
    x, w = g.uniform(-0.9, 0.9, (n, 6)), g.random((n, 6))
    return np.ascontiguousarray(np.einsum("np,npm->nm", w / w.sum(1, keepdims=True),
                                          np.cos(np.arange(M) * np.arccos(x)[..., None])))


def close(rho, ref):
    return np.max(np.abs(rho - ref) / np.max(np.abs(ref), axis=1, keepdims=True)) <= 2e-7


@pytest.mark.parametrize("n", [1, 7, 511, 512, 515])
def test_prior_rows(ctx, n):
    X = moments(n, 128, n).astype(np.float32)
    Y = np.zeros((n, kite.MLP_OUT), np.float32)
    kite.mlp_forward(ctx, np.zeros(kite.mlp_param_count(), np.float32), X, n, Y, prior=kite.jackson_prior(LO, HI))
    assert close(Y, jackson_density(X.astype(np.float64)))


@pytest.mark.parametrize("n,mu_ld,M", [(3, 128, 1), (9, 130, 2), (5, 129, 127), (2, 300, 128), (513, 140, 129),
                                       (520, 260, 257), (1, 8193, 8192), (2, 8193, 8193)])
def test_forced_fallback_rows(ctx, n, mu_ld, M):
    mu = moments(n, mu_ld, n + M)
    model = kite.model_import(ctx, np.zeros(kite.mlp_param_count(), np.float32), LO, HI)
    rho, fell, dev = np.zeros((n, kite.MLP_OUT), np.float32), np.zeros(n, np.int32), np.zeros(n)
    kite.learned_dos(ctx, model, mu, mu_ld, n, 0.0, 16, M, rho, fell, dev)
    assert np.all(fell == 1) and close(rho, jackson_density(mu[:, :M]))


@pytest.mark.parametrize("kcheck", [1, 15, 16, 17, 40])
def test_gate_orders(ctx, kcheck):
    g = np.random.Generator(np.random.PCG64(kcheck))
    rho, mu = g.random((6, kite.MLP_OUT)).astype(np.float32), g.standard_normal((6, 40)) * 0.1
    rho[3, 17] = np.inf
    flags, dev = np.zeros(6, np.int32), np.zeros(6)
    kite.learned_gate(ctx, rho, mu, 40, 6, kcheck, LO, HI, 1.0, flags, dev)
    T = np.cos(np.arange(kcheck)[:, None] * np.arccos(EPS)[None, :])
    ok = np.arange(6) != 3
    ref = np.abs(rho[ok].astype(np.float64) * 0.5 * (HI - LO) @ T.T * (2.0 / 1024) - mu[ok, :kcheck]).max(1)
    assert np.max(np.abs(dev[ok] - ref)) <= 1e-11 and np.isinf(dev[3]) and flags[3] == 1
    assert np.array_equal(flags[ok] == 1, ref > 1.0)
