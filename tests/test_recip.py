"""The quotients of the plan's factors (csrc/recip.h): a product by the reciprocal corrected by its
remainder, restated in exact rational arithmetic, rounds as a division does."""
from fractions import Fraction

import numpy as np
import pytest


def quotient(a, d):
    r = 1.0 / d
    q = a * r
    rem = float(Fraction(a) - Fraction(q) * Fraction(d))          # fma(-q, d, a)
    return float(Fraction(rem) * Fraction(r) + Fraction(q))       # fma(rem, r, q)


@pytest.mark.parametrize("spread", [0, 40, 600])
def test_corrected_quotient_is_the_rounded_one(spread):
    g = np.random.default_rng(spread)
    a = g.standard_normal(4000) * 2.0 ** g.integers(-spread, spread + 1, 4000)
    d = g.uniform(1.0, 2.0, 4000) * 2.0 ** g.integers(-spread // 2, spread // 2 + 1, 4000)
    for x, y in zip(a, d):
        assert quotient(float(x), float(y)) == float(x) / float(y)
