"""The float bin rule's filter in exact rational arithmetic: where it decides, its
cell is that of the correctly rounded double quotient."""
import random
from fractions import Fraction

import numpy as np
import pytest

F = np.float32


def add_down(a, b):
    """a + b rounded down to float."""
    exact = Fraction(float(a)) + Fraction(float(b))
    r = F(float(a) + float(b))
    return r if Fraction(float(r)) <= exact else np.nextafter(r, F(-np.inf))


def fma(a, b, c):
    exact = Fraction(float(a)) * Fraction(float(b)) + Fraction(float(c))
    lo = F(float(exact))   # double, then float: the second rounding moves it by at most one neighbour
    return min((np.nextafter(lo, F(-np.inf)), lo, np.nextafter(lo, F(np.inf))),
               key=lambda v: abs(Fraction(float(v)) - exact))


def fast(x, x0, H, nb):
    """(decided, cell) of the filter."""
    binh = F(0.5 - abs(x0 * (1.0 / H)) * 2.0**-21 - 2.0**-24)
    q = F(F(F(x) - F(x0)) * F(1.0 / H))
    y = add_down(q, F(8388608.0))
    i = int(np.float32(y).view(np.int32)) - 0x4B000000
    d = F(q - F(y - F(8388607.5)))
    return bool(abs(d) < fma(q, F(-(2.0**-21)), binh)) and 0 <= i < nb, i


@pytest.mark.parametrize("seed", range(4))
def test_decided_cells_are_the_exact_ones(seed):
    rng = random.Random(seed)
    decided = 0
    for _ in range(4000):
        nb = rng.choice([2, 3, 17, 128, 1000, 4096])
        L = rng.uniform(0.1, 5.0)
        x0 = rng.choice([0.0, rng.uniform(-10.0, 10.0), 300.0])
        H = L / nb
        k = rng.randint(-1, nb)
        near = rng.choice([0.0, 2.0**-26, 2.0**-22, 2.0**-18, 2.0**-12, 0.3]) * rng.choice([-1.0, 1.0])
        x = float(F(x0 + H * (k + near)))
        ok, i = fast(x, x0, H, nb)
        if ok:
            decided += 1
            q = (x - x0) / H
            assert i == int(np.floor(q)) and 0 <= q < nb, (x, x0, H, nb)
    assert decided > 500
