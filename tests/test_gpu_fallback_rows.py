"""The plain fallback of the learned path at the order where a single flagged row leaves the table
of Chebyshev polynomials (256), and several rows at the largest order that keeps it (8192);
bar of test_gpu_cheb_rows.py (FP32 outputs of FP64 sums: 2e-7 of the row's largest value)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

kite = pytest.importorskip("paper_1910_05194_gb300")
LO, HI = -11.0, 12.5
EPS = -1.0 + (2.0 * np.arange(1024) + 1.0) / 1024


def jackson_density(mu):
    M = mu.shape[1]
    n, q = np.arange(M), np.pi / (M + 1)
    g = ((M - n + 1) * np.cos(q * n) + np.sin(q * n) / np.tan(q)) / (M + 1) * np.where(n == 0, 1.0, 2.0)
    T = np.cos(n[:, None] * np.arccos(EPS)[None, :])
    return (mu * g) @ T / (np.pi * np.sqrt(1.0 - EPS ** 2) * 0.5 * (HI - LO))


@pytest.mark.parametrize("n,flagged,M", [(1, 1, 256), (1, 1, 257), (40, 1, 256), (40, 1, 257), (2, 2, 257), (3, 2, 8192)])
def test_flagged_rows(n, flagged, M):
    g = np.random.Generator(np.random.PCG64(n + M))
    mu_ld = max(M, 128)
    x, w = g.uniform(-0.9, 0.9, (n, 6)), g.random((n, 6))
    mu = np.ascontiguousarray(np.einsum("np,npm->nm", w / w.sum(1, keepdims=True),
                                        np.cos(np.arange(mu_ld) * np.arccos(x)[..., None])))
    mu[flagged:, :] = 0.0  # the network of zeros predicts the prior: only these rows agree
    with kite.Context(0) as ctx:
        model = kite.model_import(ctx, np.zeros(kite.mlp_param_count(), np.float32), LO, HI)
        rho, fell, dev = np.zeros((n, kite.MLP_OUT), np.float32), np.zeros(n, np.int32), np.zeros(n)
        kite.learned_dos(ctx, model, mu, mu_ld, n, 1e-6, 16, M, rho, fell, dev)
    ref = jackson_density(mu[:, :M])
    assert fell.sum() == flagged and np.all(fell[:flagged] == 1)
    assert np.all(np.abs(rho - ref)[:flagged].max(1) <= 2e-7 * np.abs(ref)[:flagged].max(1))
    assert not rho[flagged:].any()
