"""The kernels' own reciprocal and square root (``recip`` and ``root`` of ``csrc/dg_common.cuh``)
against exact results: random mantissas at every exponent, both sides of the ranges in which they
iterate, and special values, where they have to give what 1.0 / x and sqrt(x) give.

Bound: half an ulp of rounding and what the iterations leave, 2^-20 ulp (recip: e is exact to
2^-73) and less (root): 0.50001 ulp."""
import math
from fractions import Fraction as F

import numpy as np
import pytest

from paper_2409_09620_gb300 import native as N

pytestmark = pytest.mark.gpu


def _mantissas(rng, n):
    m = rng.integers(0, 1 << 52, n, dtype=np.int64)
    m[:64] = [0, 1, 2, 3, (1 << 52) - 1, (1 << 52) - 2, 1 << 51, (1 << 51) - 1] * 8
    return m


def _make(exponent_field, mantissa):
    return ((np.asarray(exponent_field, np.int64) << 52) | mantissa).view(np.float64)


def test_recip_is_within_half_an_ulp():
    rng = np.random.default_rng(1)
    n = 60000
    x = _make(rng.integers(1, 2046, n), _mantissas(rng, n)) * rng.choice([1.0, -1.0], n)
    x[:8192] = _make(rng.choice([1, 2, 3, 2042, 2043, 2044, 2045], 8192), _mantissas(rng, 8192))
    y = N.probe_math(N.MATH_RECIP, x)
    worst = F(0)
    for a, r in zip(x.tolist(), y.tolist()):
        worst = max(worst, abs(F(r) - 1 / F(a)) / F(math.ulp(r)))
    assert worst <= F(50001, 100000), float(worst)
    # correctly rounded but for the arguments whose result is within 2^-16 ulp of a midpoint
    many = _make(rng.integers(2, 2043, 1 << 20), _mantissas(rng, 1 << 20))
    assert np.mean(N.probe_math(N.MATH_RECIP, many) != 1.0 / many) < 1e-4


def test_root_is_within_half_an_ulp():
    rng = np.random.default_rng(2)
    n = 60000
    x = _make(rng.integers(1, 2047, n), _mantissas(rng, n))
    x[:8192] = _make(rng.choice([126, 127, 128, 129, 1918, 1919, 1920, 1921], 8192), _mantissas(rng, 8192))
    y = N.probe_math(N.MATH_ROOT, x)
    lim = F(50001, 100000)
    for a, r in zip(x.tolist(), y.tolist()):   # |r - sqrt(a)| <= lim ulp, squared
        u = lim * F(math.ulp(r))
        assert (F(r) - u) ** 2 <= F(a) <= (F(r) + u) ** 2, (a, r)
    many = _make(rng.integers(1, 2047, 1 << 20), _mantissas(rng, 1 << 20))
    assert np.mean(N.probe_math(N.MATH_ROOT, many) != np.sqrt(many)) < 1e-4


@pytest.mark.filterwarnings("ignore:divide by zero")
def test_special_values():
    x = np.array([0.0, -0.0, np.inf, -np.inf, np.nan, 5e-324, -5e-324, 2.0 ** -1022, 2.0 ** -1030, 2.0 ** 1023,
                  1.7976931348623157e308, -1.7976931348623157e308, 1.0, -1.0, 4.0, 3.0])
    with np.errstate(all="ignore"):
        np.testing.assert_array_equal(N.probe_math(N.MATH_RECIP, x), 1.0 / x)
        x = x[~(x < 0.0)]
        got, want = N.probe_math(N.MATH_ROOT, x), np.sqrt(x)
    np.testing.assert_array_equal(got, want)
    assert np.array_equal(np.signbit(got[:2]), [False, True])
