"""The correctly rounded quotient of the bin rule and of the FP64 weights,
a / b from y = RN(1 / b) by two residual corrections, in exact rational
arithmetic: equal to IEEE division for grid-like operands, for random ones and
next to the midpoints between two doubles."""
import math
import random
from fractions import Fraction

import numpy as np
import pytest


def fma(a, b, c):
    """RN(a b + c) through exact rationals (float() of a Fraction rounds to nearest even)."""
    return float(Fraction(a) * Fraction(b) + Fraction(c))


def quotient(a, b):
    y = 1.0 / b
    q0 = a * y
    q1 = fma(fma(-q0, b, a), y, q0)
    return fma(fma(-q1, b, a), y, q1)


@pytest.mark.parametrize("seed", range(4))
def test_equals_ieee_division(seed):
    rng = random.Random(seed)
    for _ in range(3000):
        kind = rng.randrange(4)
        if kind == 0:      # particle offsets over a bulk spacing
            b = rng.uniform(0.2, 3.0) / rng.randint(2, 400)
            a = rng.uniform(0.0, 400.0) * b
        elif kind == 1:    # next to a cell face
            b = rng.uniform(0.2, 3.0) / rng.randint(2, 400)
            a = float(np.nextafter(rng.randint(1, 400) * b, math.inf if rng.random() < 0.5 else -math.inf))
        elif kind == 2:    # any significands
            b = rng.uniform(1.0, 2.0) * 2.0 ** rng.randint(-60, 60)
            a = rng.uniform(1.0, 2.0) * 2.0 ** rng.randint(-60, 60) * rng.choice([-1.0, 1.0])
        else:              # a quotient close to the midpoint of two doubles
            b = rng.uniform(1.0, 2.0)
            q = rng.uniform(1.0, 2.0)
            a = float((Fraction(q) + Fraction(math.ulp(q)) / 2) * Fraction(b))
        assert quotient(a, b) == a / b, (a, b)
    assert quotient(0.0, 0.3) == 0.0
