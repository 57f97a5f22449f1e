"""The kernels' quotient of a chunk's weight and mass, restated: an approximate reciprocal (up to one unit in the last place off, either
way), the product, and one step on its exact remainder.  Whatever the reciprocal, the result is as close to the real quotient as a
rounded division is, to 1e-5 of a unit in the last place; without the step it is not."""
from fractions import Fraction

import numpy as np
import pytest


def rounded(x):
    """Fraction -> nearest float32 (of numbers that are not subnormal), ties to even."""
    e = 0
    while x >= 2 ** 24:
        x, e = x / 2, e + 1
    while x < 2 ** 23:
        x, e = x * 2, e - 1
    n = x.numerator // x.denominator
    rest = x - n
    n += rest > Fraction(1, 2) or (rest == Fraction(1, 2) and n % 2 == 1)
    return Fraction(n) * Fraction(2) ** e


def ulp(x):
    return Fraction(float(np.spacing(np.float32(float(x)))))


@pytest.mark.parametrize("off", [-1, 0, 1])
def test_quotient_is_as_close_as_the_rounded_division(off):
    rng = np.random.default_rng(off + 5)
    worst = plain = Fraction(0)
    for _ in range(500):
        z = Fraction(float(np.float32(np.exp(rng.uniform(0.0, np.log(64.0))))))
        w = Fraction(float(np.float32(np.exp(rng.uniform(-60.0, 16.0)))))
        r = rounded(1 / z)
        r += off * ulp(r)
        q = rounded(w * r)
        left = w - z * q
        left = (1 if left > 0 else -1) * rounded(abs(left)) if left else Fraction(0)
        got = rounded(q + left * r)
        worst = max(worst, abs(got - w / z) / ulp(w / z))
        plain = max(plain, abs(q - w / z) / ulp(w / z))
    assert worst <= Fraction(1, 2) + Fraction(1, 100000)
    assert plain > Fraction(3, 4)
