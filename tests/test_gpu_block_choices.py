"""The block of the Kubo-Greenwood sum (512 threads from 1536 orders on with at most one energy per
SM, else 256) around that line, against the definition.  Bar: a last place of theta (2^-52 each side)
moves cos(n theta) by n 2^-52 in each of the two factors, and the sums round M terms twice: 8 M 2^-53
of sum |c_n mu_nm c_m|."""
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


@pytest.mark.parametrize("M", [1535, 1536])
@pytest.mark.parametrize("K", [1, 152, 153])
def test_greenwood_blocks(ctx, M, K):
    g = np.random.Generator(np.random.PCG64(M + K))
    x = np.sort(g.uniform(-0.9, 0.9, 12))
    C = np.cos(np.arange(M)[:, None] * np.arccos(x)[None, :])
    a = g.standard_normal((12, 12)) + 1j * g.standard_normal((12, 12))
    mu = np.ascontiguousarray(C @ np.abs(a) ** 2 @ C.T / 12, dtype=np.complex128)
    E = np.linspace(-8.0, 8.5, K)
    out = np.zeros(K)
    kite.reconstruct_sigma_dc(ctx, mu, M, M, kite.HONEYCOMB, kite.KERNEL_JACKSON, 0.0, LO, HI, E, K, out)
    ref = oracle.sigma_dc(mu, E, LO, HI, oracle.HONEYCOMB)
    c = 2.0 / (np.pi * np.sqrt(1.0 - ((E - 0.5 * (HI + LO)) / (0.5 * (HI - LO))) ** 2))
    scale = np.pi * 4.0 / np.sqrt(3.0) * c ** 2 * np.abs(mu.real).sum()
    assert np.all(np.abs(out - ref) <= 8 * M * 2.0 ** -53 * scale)
