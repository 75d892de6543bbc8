"""The leader's confidence division by the patch area, checked on the CPU.

C(p) = sum / P^2 (Eq. 2) for a patch inside the image: the kernel divides by
the known P^2 with y = RN(1/P^2): q0 = RN(a y), then twice r = RN(a - q b)
(one FMA, exact), q = RN(q + r y).  After the first correction q is within an
ulp of a / b, and Markstein's theorem makes the second one the correctly
rounded quotient.  Checked against the exact quotient's rounding for every
patch size the kernel has, on sums of every binade up to P^2, on sums next to
multiples of the area, and on the smallest sums the path accepts.
"""
import random
from fractions import Fraction

import pytest


def fma(a: float, b: float, c: float) -> float:
    return float(Fraction(a) * Fraction(b) + Fraction(c))


def by_reciprocal(a: float, b: float, y: float) -> float:
    q = a * y
    q = fma(fma(-q, b, a), y, q)
    return fma(fma(-q, b, a), y, q)


@pytest.mark.parametrize("r", range(1, 9))
def test_confidence_division_is_correctly_rounded(r):
    b = float((2 * r + 1) ** 2)
    y = 1.0 / b
    rng = random.Random(r)
    sums = [rng.uniform(0.5, 1.0) * 2.0 ** rng.randint(-60, (2 * r + 1).bit_length() * 2) for _ in range(3000)]
    sums += [min(s, b) for s in sums[:200]]
    for n in range(1, int(b) + 1):
        for s in (float(n), n * b / (n + 1.0), n / 3.0):
            sums += [s, s * (1 + 2.0 ** -52), s * (1 - 2.0 ** -53)]
    sums += [1.01e-250 * rng.uniform(1, 8) for _ in range(200)]
    for a in sums:
        assert by_reciprocal(a, b, y) == a / b, (r, a)
