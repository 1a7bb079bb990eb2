"""The FP64 arithmetic on the integer pipes (products, halves, reciprocals, square roots) against exact integers.

Bounds, from the algorithms: a product keeps all bits of the 106-bit product and rounds half up, 1/2 ulp.  The
reciprocal and the reciprocal square root round once (1/2 ulp) after a correction cut at 2^-60 of a mantissa in [1, 2)
or (1/2, 1] (2^-7 ulp), a product cut 2^-10 ulp below and a cubic term below 2^-10 ulp: 0.51 ulp.  The square root is
x times that, 0.51 ulp in the wider of the two scales and another rounding: 1.53 ulp.  Outside the normal range:
subnormal operands count as zero and results below 2^-1022 are zero; the product of an infinite or NaN operand or
beyond the range is NaN; the reciprocals of zero, subnormal, infinite and NaN arguments are NaN, 1 / x for
|x| >= 2^1022 is zero, 1 / sqrt(x) and sqrt(x) of negative arguments NaN, sqrt(+0) zero."""
import itertools
import math
from fractions import Fraction

import numpy as np
import pytest

from paper_1912_11908_gb300 import workloads as W  # noqa: F401
from test_gpu_flow3d import ibm  # noqa: F401  (fixture)

pytestmark = pytest.mark.gpu

TINY, HUGE = Fraction(1, 1 << 1022), Fraction(1 << 1024)
ONES = float.fromhex("0x1.fffffffffffffp0")


def _edges():
    m = [1.0, 1.0 + 2.0 ** -52, 1.5, ONES, 1.0 + 2.0 ** -26, 4.0 / 3.0]
    e = [-1022, -1021, -1020, -512, -511, -2, -1, 0, 1, 2, 510, 511, 512, 1020, 1021, 1022, 1023]
    v = [0.0, 5e-324, math.ldexp(ONES, -1023), math.inf, math.nan] + [math.ldexp(x, k) for x in m for k in e]
    return np.array(v + [-x for x in v])


def _random(n, lo, hi, seed):
    rng = np.random.default_rng(seed)
    x = np.ldexp(1.0 + rng.integers(0, 1 << 52, n) * 2.0 ** -52, rng.integers(lo, hi, n))
    return x * rng.choice([-1.0, 1.0], n)


def _normal(x):
    return math.isfinite(x) and abs(x) >= 2.0 ** -1022


def _ulp(f):
    """The spacing of doubles at the positive fraction f."""
    k = f.numerator.bit_length() - f.denominator.bit_length()
    if f < (Fraction(1 << k) if k >= 0 else Fraction(1, 1 << -k)):
        k -= 1
    k = max(k, -1022) - 52
    return Fraction(1 << k) if k >= 0 else Fraction(1, 1 << -k)


def _product_ok(a, b, got):
    if not (math.isfinite(a) and math.isfinite(b)):
        return math.isnan(got)
    if not (_normal(a) and _normal(b)):
        return got == 0.0
    p = Fraction(a) * Fraction(b)
    if abs(p) >= HUGE - Fraction(1 << 970):  # rounds beyond the largest double
        return math.isnan(got) or math.isinf(got)
    if abs(p) < TINY:
        return got == 0.0 or abs(Fraction(got)) == TINY
    return math.isfinite(got) and abs(Fraction(got) - p) * 2 <= _ulp(abs(p))


def test_products(ibm):  # noqa: F811
    e = _edges()
    pairs = np.array(list(itertools.product(e, e)))
    a = np.concatenate([pairs[:, 0], _random(60000, -500, 500, 1), _random(20000, -1022, 1024, 2),
                        _random(20000, 0, 1, 3)])
    b = np.concatenate([pairs[:, 1], _random(60000, -500, 500, 4), _random(20000, -1022, 1024, 5),
                        _random(20000, 0, 1, 6)])
    # products of 54 bits: exact ties
    n = 20000
    rng = np.random.default_rng(7)
    a = np.concatenate([a, rng.integers(1 << 26, 1 << 27, n) | 1]).astype(np.float64)
    b = np.concatenate([b, rng.integers(1 << 26, 1 << 27, n) | 1]).astype(np.float64)
    out = ibm.fp64_arithmetic(ibm.FP64_MUL, a, b)
    bad = [(x, y, z) for x, y, z in zip(a.tolist(), b.tolist(), out.tolist()) if not _product_ok(x, y, z)]
    assert not bad, (len(bad), bad[:5])


def test_halves(ibm):  # noqa: F811
    x = np.concatenate([_edges(), _random(20000, -1022, 1024, 8)])
    got = ibm.fp64_arithmetic(ibm.FP64_HALF, x)
    want = np.where(np.abs(x) < 2.0 ** -1021, np.copysign(0.0, x), 0.5 * x)
    np.testing.assert_array_equal(got, want)


def _worst(x, got, ok, error):
    """Largest error in ulps over the arguments in range, and the arguments of a wrong special value."""
    worst, bad = 0.0, []
    for a, z in zip(x.tolist(), got.tolist()):
        special = ok(a)
        if special is not None:
            if not (math.isnan(z) if math.isnan(special) else z == special):
                bad.append((a, z))
        elif not _normal(z):
            bad.append((a, z))
        else:
            worst = max(worst, error(a, z))
    return worst, bad


def test_reciprocals(ibm):  # noqa: F811
    x = np.concatenate([_edges(), _random(60000, -1022, 1024, 9), _random(60000, 0, 1, 10)])

    def special(a):
        if not _normal(a):
            return math.nan
        return math.copysign(0.0, a) if abs(a) >= 2.0 ** 1022 else None

    def error(a, z):
        f = 1 / Fraction(a)
        return float(abs(Fraction(z) - f) / _ulp(abs(f)))

    worst, bad = _worst(x, ibm.fp64_arithmetic(ibm.FP64_RCP, x), special, error)
    print("1 / x: %.4f ulp" % worst)
    assert not bad and worst <= 0.51, (worst, bad[:5])


def _root(f):
    """sqrt of a positive fraction to 2^-90 relative."""
    s = 1 << (2 * max(0, 110 - (f.numerator.bit_length() - f.denominator.bit_length()) // 2))
    return Fraction(math.isqrt(f.numerator * s // f.denominator), math.isqrt(s))


@pytest.mark.parametrize("op", ["FP64_RSQRT", "FP64_SQRT"])
def test_square_roots(ibm, op):  # noqa: F811
    x = np.concatenate([_edges(), np.abs(_random(40000, -1022, 1024, 11)), np.abs(_random(40000, 0, 2, 12))])

    def special(a):
        if _normal(a) and a > 0.0:
            return None
        return 0.0 if op == "FP64_SQRT" and math.copysign(1.0, a) > 0.0 and a < 1.0 else math.nan

    def error(a, z):
        f = _root(Fraction(a))
        f = f if op == "FP64_SQRT" else 1 / f
        return float(abs(Fraction(z) - f) / _ulp(f))

    worst, bad = _worst(x, ibm.fp64_arithmetic(getattr(ibm, op), x), special, error)
    print("%s: %.4f ulp" % (op, worst))
    assert not bad and worst <= (0.51 if op == "FP64_RSQRT" else 1.53), (worst, bad[:5])


def test_bad_arguments_are_refused(ibm):  # noqa: F811
    with pytest.raises(ibm.IbmError):
        ibm.fp64_arithmetic(5, np.ones(3))
    with pytest.raises(ibm.IbmError):
        ibm.fp64_arithmetic(ibm.FP64_MUL, np.ones(3))
