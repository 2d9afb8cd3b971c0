"""The quotient of the treecode series (csrc/farfield.cu, TcDiv): q = a y with y = 1 / b, then twice
q + y (a - b q) with fused operations, restated in exact arithmetic with one rounding per operation, against
the correctly rounded a / b: equal down to |a| = 2^-102 in FP32 and 2^-969 in FP64, within an ulp below."""
import random
from fractions import Fraction

import pytest


def rounded(x, bits, emin):
    """x to the nearest number of `bits` significant bits and least exponent emin (ties to even)."""
    if x == 0:
        return Fraction(0)
    n, m = abs(x).numerator.bit_length(), x.denominator.bit_length()
    e = n - m  # 2^(e-1) < |x| < 2^(e+1)
    if abs(x) < Fraction(2) ** e:
        e -= 1
    ulp = Fraction(2) ** (max(e, emin) - bits + 1)
    return round(x / ulp) * ulp  # (Python rounds half to even)


@pytest.mark.parametrize("bits,emin,low", [(24, -126, -102), (53, -1022, -969)])
def test_quotient_is_correctly_rounded(bits, emin, low):
    rng = random.Random(5)

    def r(x):
        return rounded(x, bits, emin)

    def number(lo, hi):
        return Fraction(rng.getrandbits(bits) | 1 << (bits - 1)) * Fraction(2) ** (rng.randint(lo, hi) - bits + 1) * rng.choice((1, -1))

    def quotient(a, b):
        y = r(1 / b)
        q = r(a * y)
        for _ in range(2):
            q = r(q + y * r(a - b * q))
        return q

    for _ in range(4000):
        a, b = number(low, 20), abs(number(-10, 24))
        if abs(a / b) >= Fraction(2) ** emin:
            assert quotient(a, b) == r(a / b)
    for _ in range(2000):  # below the range: within an ulp
        a, b = number(emin, low - 1), abs(number(-10, 24))
        ulp = Fraction(2) ** (emin - bits + 1)
        assert abs(quotient(a, b) - a / b) <= max(ulp, abs(a / b) * Fraction(2) ** (1 - bits))
