"""The two-limb integer arithmetic of the FP64 Gram-Schmidt (csrc/fixed.cuh), replayed with Python's exact
integers: the limbs' error, and that 64 products never overflow a 64-bit sum."""
import math
import random
from fractions import Fraction

import pytest

LIM = 1 << 63


def limbs(x, e):
    """(h, l) of x on the scale 2^e: the magnitude truncated to 55 bits with a one below, two's complement."""
    if x == 0.0:
        return 0, 0
    f = 2 * int(abs(Fraction(x)) * Fraction(2) ** (55 - e)) + 1
    f = -f if x < 0 else f
    return f >> 28, f & ((1 << 28) - 1)


def stored(x, e):
    """The basis form: x 2^(60 - e) rounded to nearest."""
    q = Fraction(x) * Fraction(2) ** (60 - e)
    f = math.floor(abs(q) + Fraction(1, 2))
    return -f if q < 0 else f


def rounded(F):
    F += 8
    return F >> 32, (F & 0xffffffff) >> 4


@pytest.mark.parametrize("e", [-900, -7, 0, 40])
def test_limb_errors_and_sum(e):
    rng = random.Random(e)
    xs = [math.ldexp(rng.uniform(-1, 1) * 2.0 ** -rng.choice([0, 0, 3, 9, 30, 70]), e) for _ in range(64)] + [0.0]
    ys = [rng.gauss(0, 0.2) for _ in range(65)]
    ys = [max(-0.999, min(0.999, y)) for y in ys]
    H = M = L = 0
    for x, y in zip(xs[:64], ys):
        (h, l), (p, q) = rounded(stored(x, e)), limbs(y, 0)
        assert abs(h) <= 1 << 28 and 0 <= l < 1 << 28 and abs(p) <= 1 << 28 and 0 <= q < 1 << 28
        assert abs(Fraction(h * 2 ** 28 + l) * Fraction(2) ** (e - 56) - Fraction(x)) <= Fraction(2) ** (e - 57) * (1 + Fraction(1, 8))
        assert abs(Fraction(p * 2 ** 28 + q, 2 ** 56) - Fraction(y)) <= Fraction(1, 2 ** 56)
        H, M, L = H + h * p, M + h * q + l * p, L + l * q
    total = (H * 2 ** 56 + M * 2 ** 28 + L) * Fraction(2) ** (e - 112)
    exact = sum(Fraction(x) * Fraction(y) for x, y in zip(xs[:64], ys))
    # each factor off by 2^-57 (1 + 1/8) or 2^-56 of its scale, the other below 1: 64 (2^-57 9/8 + 2^-56) 2^e and a margin
    assert abs(total - exact) <= 64 * Fraction(2) ** (e - 55)
    assert stored(math.ldexp(0.75, e), e) == 3 << 58 and limbs(0.0, 0) == (0, 0)


def test_sums_cannot_overflow():
    top, low = 1 << 28, (1 << 28) - 1
    assert 64 * top * top < LIM and 64 * 2 * top * low < LIM and 64 * low * low < LIM
    # the small columns of the update: 28 by 22 bits, 4 (m + 1) products, m <= 1023
    assert 4 * 1024 * top * (1 << 22) <= LIM
