"""The conductivity reconstructions at the orders where their cosine sums change path: dense
FP64 products below M = 64 and above 2048, the non-uniform transform between, with its grid
sizes (powers of two) and odd orders and node counts.  Against the oracle's direct sums at
the bars of test_gpu_sigma.py and test_gpu_hall.py (1e-9 and 1e-10 of the largest value: the
errors of either path, about M * 2^-53 per cosine sum, lie four orders below)."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

kite = pytest.importorskip("paper_1910_05194_gb300")
LO, HI = -8.7, 9.1  # an asymmetric window: de_plus != 0


@pytest.fixture(scope="module")
def ctx():
    c = kite.Context(0)
    yield c
    c.close()


def moments(M, seed, hermitian):
    """mu_nm of a small random model (hermitian: alpha = beta), and of a non-Hermitian family
    pair otherwise."""
    g = np.random.Generator(np.random.PCG64(seed))
    x = np.sort(g.uniform(-0.9, 0.9, 12))
    C = np.cos(np.arange(M)[:, None] * np.arccos(x)[None, :])
    a = g.standard_normal((12, 12)) + 1j * g.standard_normal((12, 12))
    return np.ascontiguousarray(C @ (np.abs(a) ** 2 if hermitian else a) @ C.T / 12, dtype=np.complex128)


@pytest.mark.parametrize("M,n_quad,K,kT", [(63, 0, 3, 0.0), (64, 0, 5, 0.0), (65, 31, 1, 0.05), (128, 129, 4, 0.0),
                                           (201, 0, 6, 0.02), (513, 300, 2, 0.0), (1, 8, 2, 0.0)])
def test_optical_conductivity_across_the_orders(ctx, M, n_quad, K, kT):
    mu = moments(M, M, True)
    om = np.linspace(0.3, 9.0, K)
    out = np.zeros(K, np.complex128)
    kite.reconstruct_sigma(ctx, mu, M, M, kite.HONEYCOMB, kite.KERNEL_JACKSON, LO, HI, 0.4, kT, 0.2, om, K, out, n_quad)
    ref = oracle.sigma_xx(mu, om, LO, HI, 0.4, 0.2, 0, kernel="jackson", kT=kT, n_quad=n_quad or 2 * M + 64)
    assert np.max(np.abs(out - ref)) <= 1e-9 * np.max(np.abs(ref))


@pytest.mark.parametrize("M,n_quad,K,kT", [(63, 0, 2, 0.0), (64, 0, 3, 0.03), (65, 77, 5, 0.0), (150, 0, 4, 0.0),
                                           (257, 201, 2, 0.0), (600, 128, 1, 0.0), (2, 9, 3, 0.0)])
def test_bastin_conductivity_across_the_orders(ctx, M, n_quad, K, kT):
    mu = moments(M, M + 1, False)
    E = np.linspace(-5.0, 6.0, K)
    out = np.zeros(K)
    kite.reconstruct_sigma_dc_bastin(ctx, mu, M, M, kite.SQUARE, kite.KERNEL_LORENTZ, 3.0, LO, HI, 0.3, kT, E, K, out,
                                     n_quad)
    ref = oracle.sigma_dc_bastin(mu, E, LO, HI, 0.3, 1, kernel="lorentz", lam=3.0, kT=kT, n_quad=n_quad or 2 * M + 64)
    assert np.max(np.abs(out - ref)) <= 1e-10 * max(1.0, np.max(np.abs(ref)))
