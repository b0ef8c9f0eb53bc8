"""The Gauss-Legendre weights behind the optical sums, from the host (up to 64 nodes) and from the
device: one moment and a smooth integrand (kT = 2 eV, eta = 2 eV), against a rule and sums in extended
precision.  A weight is rounded by a few 2^-53, with either sign, and so is the sum of a rule
(4e-16 of it at most, measured on the rule alone); a last Newton step that is not allowed for
makes every weight too large, by 1 to 3e-15 of the sum.  So the mean deviation over several rules
stays below 6e-16, a single one below 2e-15."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

kite = pytest.importorskip("paper_1910_05194_gb300")
L = np.longdouble
PI = L("3.14159265358979323846264338327950288")


def gauss(K):
    x = np.polynomial.legendre.leggauss(K)[0].astype(L)
    for _ in range(3):
        p0, p1 = np.ones_like(x), x.copy()
        for j in range(2, K + 1):
            p0, p1 = p1, ((2 * j - 1) * x * p1 - (j - 1) * p0) / L(j)
        dp = K * (x * p1 - p0) / (x * x - 1)
        x = x - p1 / dp
    p0, p1 = np.ones_like(x), x.copy()
    for j in range(2, K + 1):
        p0, p1 = p1, ((2 * j - 1) * x * p1 - (j - 1) * p0) / L(j)
    dp = K * (x * p1 - p0) / (x * x - 1)
    return x, 2 / ((1 - x * x) * dp * dp)


def exact(om, lo, hi, EF, eta, kT, K):
    minus, plus = L(0.5 * (hi - lo)), L(0.5 * (hi + lo))
    x, w = gauss(K)
    e = np.cos(PI * (x + 1) / 2)
    D = w / (1 + np.exp((e * minus + plus - L(EF)) / L(kT)))  # (2/pi) cos(0) times pi/2
    wv, et = L(om) / minus, L(eta) / minus
    r = np.sqrt(1 - (e + wv + 1j * et) ** 2)
    a = np.sqrt(1 - (e - wv - 1j * et) ** 2)
    s = ((-2j / r + 2j / a) * D).sum() * (-L(1) / 4)
    return -1j * 4 / np.sqrt(L(3)) / wv * s


@pytest.mark.parametrize("rules", [range(12, 65, 4), range(66, 194, 8), range(194, 600, 34)])
def test_weights(rules):
    om = np.array([1.0, 5.0])
    dev = []
    with kite.Context(0) as ctx:
        for K in rules:
            out = np.zeros(2, np.complex128)
            kite.reconstruct_sigma(ctx, np.ones((1, 1), np.complex128), 1, 1, kite.HONEYCOMB, kite.KERNEL_NONE, -8.0, 8.0,
                                   0.0, 2.0, 2.0, om, 2, out, K)
            ref = [exact(o, -8.0, 8.0, 0.0, 2.0, 2.0, K) for o in om]
            dev.append([float(((v - r) / abs(r) * abs(r) / r).real) for v, r in zip(out, ref)])
    dev = np.array(dev)
    assert np.max(np.abs(dev)) <= 2e-15 and np.all(np.abs(dev.mean(0)) <= 6e-16)
