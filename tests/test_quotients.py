"""The kernels' quotients from a shared reciprocal: q = RN(a y), r = RN(a - b q), RN(q + r y) with
y = RN(1 / b).  The estimate q can be 1.5 units in the last place off a / b (where a's mantissa is
below b's), more than the one unit for which the textbook theorem states that the result is the
rounded quotient; here the steps are followed exactly, for every pair of mantissas at small
precisions and for FP64 and FP32 operands."""
from fractions import Fraction

import numpy as np
import pytest


def _round(x, p):
    """x to p bits, to nearest even (exact while x holds no more than 53 bits)."""
    m, e = np.frexp(x)
    return np.ldexp(np.rint(np.ldexp(m, p)), e - p)


@pytest.mark.parametrize("p", [3, 5, 8, 10, 11])
def test_every_pair_of_mantissas(p):
    n = 1 << (p - 1)
    a = np.arange(n, 2 * n, dtype=np.float64)
    far = 0
    for b in range(n, 2 * n):
        y = _round(np.float64(1.0) / b, p)
        q = _round(a * y, p)
        r = _round(a - b * q, p)
        z = _round(q + r * y, p)
        assert np.array_equal(z, _round(a / b, p)), b
        e = np.frexp(a / b)[1]
        far += int((np.abs(q - a / b) > np.ldexp(1.0, e - p)).sum())
    assert far > 0                 # the estimates the theorem leaves out do occur


def _fma(a, b, c, real):
    """a b + c rounded once."""
    v = Fraction(float(a)) * Fraction(float(b)) + Fraction(float(c))
    if real is np.float64:
        return np.float64(float(v))
    x = np.float32(float(v))       # to 24 bits: the neighbours decide, ties to even
    best = None
    for w in (np.nextafter(x, np.float32(-np.inf)), x, np.nextafter(x, np.float32(np.inf))):
        k = (abs(Fraction(float(w)) - v), int(w.view(np.uint32)) & 1)
        if best is None or k < best[0]:
            best = (k, w)
    return best[1]


@pytest.mark.parametrize("real", [np.float64, np.float32])
def test_operands_of_both_precisions(real):
    """Random operands, and pairs just below 2 with a < b, where the estimate is farthest off."""
    rng = np.random.default_rng(11)
    bits = 53 if real is np.float64 else 24
    n = 1500
    a = rng.uniform(1, 2, n) * 2.0 ** rng.integers(-20, 21, n)
    b = rng.uniform(1, 2, n) * 2.0 ** rng.integers(-20, 21, n)
    d = rng.integers(2, 3000, n)
    a2 = 2.0 - (d + rng.integers(1, 3000, n)) * 2.0 ** (1 - bits)
    b2 = 2.0 - d * 2.0 ** (1 - bits)
    for x, w in zip(np.concatenate([a, a2]).astype(real), np.concatenate([b, b2]).astype(real)):
        y = real(1.0) / w
        q = x * y
        z = _fma(_fma(-q, w, x, real), y, q, real)
        assert z == x / w, (float(x).hex(), float(w).hex())
