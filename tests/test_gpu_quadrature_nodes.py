"""The conductivity reconstructions on both sides of the number of quadrature nodes where their
cosine sums change path (dense products below 65 nodes in the optical sums, below 129 nodes of
one energy and 257 of all in Bastin's) and the rule moves from the host to the device (65
nodes), against the oracle's direct sums at the bars of
test_gpu_sigma.py and test_gpu_hall.py (1e-9 and 1e-10 of the largest value)."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

kite = pytest.importorskip("paper_1910_05194_gb300")
LO, HI = -8.7, 9.1


@pytest.fixture(scope="module")
def ctx():
    c = kite.Context(0)
    yield c
    c.close()


def moments(M, seed, hermitian):
    g = np.random.Generator(np.random.PCG64(seed))
    x = np.sort(g.uniform(-0.9, 0.9, 12))
    C = np.cos(np.arange(M)[:, None] * np.arccos(x)[None, :])
    a = g.standard_normal((12, 12)) + 1j * g.standard_normal((12, 12))
    return np.ascontiguousarray(C @ (np.abs(a) ** 2 if hermitian else a) @ C.T / 12, dtype=np.complex128)


@pytest.mark.parametrize("M", [64, 100, 321])
@pytest.mark.parametrize("n_quad,kT", [(1, 0.0), (2, 0.05), (17, 0.0), (63, 0.0), (64, 0.0), (64, 0.05), (65, 0.0), (66, 0.05)])
def test_optical_conductivity_with_few_nodes(ctx, M, n_quad, kT):
    mu, om = moments(M, M, True), np.linspace(0.3, 9.0, 5)
    out = np.zeros(5, np.complex128)
    kite.reconstruct_sigma(ctx, mu, M, M, kite.HONEYCOMB, kite.KERNEL_JACKSON, LO, HI, 0.4, kT, 0.2, om, 5, out, n_quad)
    ref = oracle.sigma_xx(mu, om, LO, HI, 0.4, 0.2, 0, kernel="jackson", kT=kT, n_quad=n_quad)
    assert np.max(np.abs(out - ref)) <= 1e-9 * np.max(np.abs(ref))


@pytest.mark.parametrize("M", [64, 100, 321])
@pytest.mark.parametrize("n_quad,K,kT", [(1, 1, 0.0), (1, 3, 0.05), (3, 5, 0.0), (128, 1, 0.0), (128, 2, 0.05), (64, 4, 0.0),
                                         (129, 1, 0.0), (129, 2, 0.0), (128, 3, 0.0), (65, 4, 0.05), (51, 5, 0.0), (52, 5, 0.0)])
def test_bastin_conductivity_with_few_nodes(ctx, M, n_quad, K, kT):
    mu, E = moments(M, M + 1, False), np.linspace(-5.0, 6.0, K)
    out = np.zeros(K)
    kite.reconstruct_sigma_dc_bastin(ctx, mu, M, M, kite.SQUARE, kite.KERNEL_LORENTZ, 3.0, LO, HI, 0.3, kT, E, K, out,
                                     n_quad)
    ref = oracle.sigma_dc_bastin(mu, E, LO, HI, 0.3, 1, kernel="lorentz", lam=3.0, kT=kT, n_quad=n_quad)
    assert np.max(np.abs(out - ref)) <= 1e-10 * max(1.0, np.max(np.abs(ref)))


@pytest.mark.parametrize("M,n_quad", [(2047, 70), (2048, 65), (2048, 64), (2049, 70), (256, 333), (257, 333)])
def test_optical_conductivity_at_the_transforms_edges(ctx, M, n_quad):
    """The largest order of the transform (8192 grid points, 128 KB of shared memory a row), the
    dense products above it, and the orders between which the grid gets coarser (256, 257)."""
    mu, om = moments(M, M, True), np.linspace(0.3, 9.0, 2)
    out = np.zeros(2, np.complex128)
    kite.reconstruct_sigma(ctx, mu, M, M, kite.HONEYCOMB, kite.KERNEL_JACKSON, LO, HI, 0.4, 0.0, 0.2, om, 2, out, n_quad)
    ref = oracle.sigma_xx(mu, om, LO, HI, 0.4, 0.2, 0, kernel="jackson", n_quad=n_quad)
    assert np.max(np.abs(out - ref)) <= 1e-9 * np.max(np.abs(ref))


@pytest.mark.parametrize("M,n_quad", [(2047, 140), (2048, 129), (2048, 128), (2049, 140), (256, 333), (257, 333)])
def test_bastin_conductivity_at_the_transforms_edges(ctx, M, n_quad):
    mu, E = moments(M, M + 1, False), np.array([1.3])
    out = np.zeros(1)
    kite.reconstruct_sigma_dc_bastin(ctx, mu, M, M, kite.SQUARE, kite.KERNEL_LORENTZ, 3.0, LO, HI, 0.3, 0.0, E, 1, out,
                                     n_quad)
    ref = oracle.sigma_dc_bastin(mu, E, LO, HI, 0.3, 1, kernel="lorentz", lam=3.0, n_quad=n_quad)
    assert np.max(np.abs(out - ref)) <= 1e-10 * max(1.0, np.max(np.abs(ref)))
