"""The bin integral over bin centres (csrc/gsn_pair64.cu): h sum_m c_m f(x + m h), |m| <= 16, c from
(delta / 2) / asinh(delta / 2), against 40-digit integrals at the rule's limits (a Gaussian of six bins, a gamma of shape 20)."""
from fractions import Fraction as Fr
from math import comb

import pytest

mp = pytest.importorskip("mpmath")
FM = 16


def coefficients():
    a = [Fr((-1) ** n * comb(2 * n, n), 4 ** n * (2 * n + 1)) for n in range(FM + 1)]   # asinh(y) / y in y^2
    b = [Fr(1)]
    for n in range(1, FM + 1):
        b.append(-sum(a[k] * b[n - k] for k in range(1, n + 1)))
    return [sum(b[n] / 4 ** n * (-1) ** (n - m) * comb(2 * n, n - m) for n in range(m, FM + 1)) for m in range(FM + 1)]


def rule(f, x):
    c = [mp.mpf(v.numerator) / v.denominator for v in coefficients()]
    return c[0] * f(x) + sum(c[m] * (f(x + m) + f(x - m)) for m in range(1, FM + 1))


@pytest.mark.parametrize("z", [0, 2, 4, 6, 8])
def test_gaussian_of_six_bins(z):
    with mp.workdps(40):
        s = mp.mpf(6)
        f = lambda x: mp.exp(-x * x / (2 * s * s))
        x = z * s + mp.mpf("0.3")
        exact = s * mp.sqrt(mp.pi / 2) * (mp.erfc((x - 0.5) / s / mp.sqrt(2)) - mp.erfc((x + 0.5) / s / mp.sqrt(2)))
        assert abs(rule(f, x) / exact - 1) < 1e-13


@pytest.mark.parametrize("x", [16.5, 20.5, 30.5, 45.5, 70.5])
def test_gamma_of_shape_twenty(x):
    with mp.workdps(40):
        mu, d = mp.mpf(30), mp.mpf(20)
        f = lambda y: mp.exp((d - 1) * mp.log(y / mu) - d * (y - mu) / mu)
        exact = mp.quad(f, [mp.mpf(x) - 0.5, x, mp.mpf(x) + 0.5])
        assert abs(rule(f, mp.mpf(x)) / exact - 1) < 1e-13
