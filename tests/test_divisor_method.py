"""The three-operation division by a fixed divisor that the FP64 kernels use for dx, restated
in exact rational arithmetic: q0 = RN(a y), y = RN(1 / b), then RN(q0 + RN(a - q0 b) y) is the
correctly rounded a / b wherever |y b - 1| <= 2^-54 (elsewhere the kernels divide)."""
import random
from fractions import Fraction

import pytest


def fma(a, b, c):
    return float(Fraction(a) * Fraction(b) + Fraction(c))          # one rounding, to nearest even


@pytest.mark.parametrize("b", [1.0, 2.0, 3.0, 5.0, 10.0, 0.3, 7.0, 12.7, 33.3, 90.0, 1000.0])
def test_three_operations_round_correctly(b):
    y = 1.0 / b
    if abs(fma(y, b, -1.0)) > 2.0 ** -54:
        pytest.skip("divided")
    rng = random.Random(int(b * 1000))
    for k in range(4000):
        m = rng.getrandbits(53)
        if k % 4 == 0:
            m &= 0xff                                              # few digits: exact quotients and ties
        if k % 4 == 1:
            m |= ((1 << 53) - 1) ^ 0xff                            # just below a power of two
        a = float(m) * 2.0 ** rng.randint(-640, 530) * rng.choice((-1, 1))
        if k % 4 == 2:                                             # next to a multiple of b
            a = float(m) * 2.0 ** -30 * b * rng.choice((1.0, 1 + 2.0 ** -52, 1 - 2.0 ** -53))
        q0 = a * y
        assert fma(fma(-q0, b, a), y, q0) == a / b, (a, b)
