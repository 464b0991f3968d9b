"""The FP64 step divides by its constants c_s^2 and c_s^4 with one product and
one fused multiply-add, m x + (x m 2^-54) for 1/c = m (1 + 2^-54 ...).  The quotients
that lie closest to a rounding boundary are those with 2 x 2^k = (2 q + 1) c + r on
the integer mantissas and a small r; every x with |r| <= R and random ones are
rounded as the exact quotient (rational arithmetic, no device)."""
import random
from fractions import Fraction as F

import pytest

CS2 = 1.0 / 3.0
R = 1201


def rn(v):
    """A rational rounded to the nearest double (ties to even)."""
    return v.numerator / v.denominator


def two_op(x, m):
    return rn(F(m) * F(x) + F(rn(F(x) * F(m * 2.0 ** -54))))


def hard_cases(c):
    ci = int(F(c) * 2 ** 60)  # the integer mantissa (trailing zeros only add exact cases)
    while ci % 2 == 0:
        ci //= 2
    while ci < 1 << 52:
        ci *= 2
    odd, tz = ci, 0
    while odd % 2 == 0:
        odd, tz = odd // 2, tz + 1
    for j in (52, 53):
        mod = 1 << (j + 1 - tz)
        inv = pow(odd, -1, mod)
        for r in range(-R, R + 1):
            if r == 0:
                continue
            q2 = (-r * inv) % mod
            while q2 < 1 << 54:
                if q2 % 2 and q2 > 1 << 53:
                    x, rest = divmod(q2 * odd + r, mod)
                    if rest == 0 and 1 << 52 <= x < 1 << 53:
                        yield float(x)
                q2 += mod


@pytest.mark.parametrize("c,m,halves", [(CS2, 3.0, 1), (CS2, 1.5, 2), (CS2 * CS2, 9.0, 1), (CS2 * CS2, 4.5, 2)])
def test_two_operation_division_rounds_correctly(c, m, halves):
    rng = random.Random(7)
    cases = list(hard_cases(c)) + [float(rng.getrandbits(52) | 1 << 52) for _ in range(20000)]
    assert len(cases) > 20500
    for x in cases:
        assert two_op(x, m) == rn(F(x) / (halves * F(c)))
        assert two_op(-x, m) == -two_op(x, m)
