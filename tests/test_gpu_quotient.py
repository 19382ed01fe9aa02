"""The quotient z / h_{j+1,j} of the Gram-Schmidt kernels (reciprocal, product, one
correction) against exact arithmetic, and against division where it divides.

The bound: with unit roundoff u, the reciprocal, the product and the residual are
each rounded once, so the sum that is rounded last is off by (2 u)(2 u) |a / h| at
most, which is 4 u units in the last place; with the last rounding 1/2 + 4 u.  For
fp32 the residual q h - a is exact in fp64; for fp64 it is formed in fractions."""
from fractions import Fraction

import numpy as np
import pytest

from gpu_helpers import dev, host, lib

pytestmark = pytest.mark.gpu


def _quot(a, h):
    return host(lib().probe_quotients(dev(a), dev(h)))


def _operands(dtype, n, e_a, e_h, seed):
    """Signed a and positive h with uniform exponents, a third each of uniform mantissas, just above a
    power of two, and just below one."""
    rng = np.random.default_rng(seed)
    eps = np.finfo(dtype).eps

    def mantissa():
        m = rng.uniform(1.0, 2.0, n).astype(dtype)
        k = rng.integers(1, 40, n)
        kind = rng.integers(0, 3, n)
        return np.where(kind == 0, m, np.where(kind == 1, 1 + k * eps, 2 - k * eps)).astype(dtype)

    a = np.ldexp(mantissa(), rng.integers(e_a[0], e_a[1], n)) * rng.choice([-1, 1], n)
    return a.astype(dtype), np.ldexp(mantissa(), rng.integers(e_h[0], e_h[1], n)).astype(dtype)


@pytest.mark.parametrize("e_a,e_h", [((-30, 1), (-5, 5)), ((-76, 76), (-49, 49))], ids=["usual", "whole range"])
def test_fp32_within_the_bound(e_a, e_h):
    a, h = _operands(np.float32, 2_000_000, e_a, e_h, 1)
    q = _quot(a, h)
    err = np.abs(q.astype(np.float64) * h - a) / (np.spacing(np.abs(q)).astype(np.float64) * h)
    assert err.max() <= 0.5 + 2.0 ** -22
    assert (q == a / h).mean() > 0.99999


@pytest.mark.parametrize("e_a,e_h", [((-60, 1), (-5, 5)), ((-680, 680), (-332, 332))], ids=["usual", "whole range"])
def test_fp64_within_the_bound(e_a, e_h):
    a, h = _operands(np.float64, 20_000, e_a, e_h, 2)
    q = _quot(a, h)
    bound = Fraction(1, 2) + Fraction(1, 2 ** 51)
    for x, y, z in zip(a.tolist(), h.tolist(), q.tolist()):
        assert abs(Fraction(z) * Fraction(y) - Fraction(x)) <= bound * Fraction(float(np.spacing(abs(z)))) * Fraction(y)
    a, h = _operands(np.float64, 2_000_000, e_a, e_h, 3)
    assert (_quot(a, h) == a / h).mean() > 0.99999


@pytest.mark.parametrize("dtype", [np.float32, np.float64])
def test_divides_outside_its_range(dtype):
    """Small and large a (subnormal residuals and quotients among them), zeros, infinities and NaN, and h
    at and beyond the limits: the division's own result."""
    f = np.finfo(dtype)
    lo, hi, big = (-149, -76, 1e15) if dtype == np.float32 else (-1074, -680, 1e100)
    small, h = _operands(dtype, 200_000, (lo, hi), (-40, 40), 4)
    large = _operands(dtype, 200_000, (-hi, f.maxexp - 42), (-40, 40), 5)[0]
    any_a = _operands(dtype, 200_000, (-60, 60), (0, 1), 6)[0]
    edge = np.resize(np.array([big, 1 / big, f.tiny, f.max, np.nextafter(dtype(big), dtype(np.inf)),
                               np.nextafter(dtype(1 / big), dtype(0)), f.tiny / 4], dtype), 200_000)
    zeros = np.resize(np.array([0.0, -0.0], dtype), 200_000)
    odd = np.resize(np.array([np.inf, -np.inf, np.nan, f.tiny, f.tiny / 2], dtype), 200_000)
    with np.errstate(all="ignore"):
        for x, y in [(small, h), (large, h), (any_a, edge), (zeros, h), (odd, h)]:
            q = _quot(x, y)
            assert np.array_equal(q, x / y, equal_nan=True)
            assert np.array_equal(np.signbit(q) | np.isnan(q), np.signbit(x / y) | np.isnan(q))
