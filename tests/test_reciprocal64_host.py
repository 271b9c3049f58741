"""The float64 reciprocal and quotient of the kernels, emulated exactly in rationals: two
Newton-Raphson steps from an approximation within 2^-19 of the true value."""
from fractions import Fraction as Fr

import numpy as np
import pytest


def fma(a, b, c):
    return float(Fr(a) * Fr(b) + Fr(c))


@pytest.mark.parametrize("err", [-2.0 ** -19, -2.0 ** -22, 0.0, 2.0 ** -19])
def test_reciprocal_and_quotient_within_half_an_ulp_and_a_hundredth(err):
    rng = np.random.default_rng(5)
    for x in np.exp(rng.uniform(np.log(1e-12), np.log(1e12), 400)):
        x, a = float(x), float(rng.uniform(-1, 1))
        r = float(1 / Fr(x) * (1 + Fr(err)))
        r = fma(r, fma(-x, r, 1.0), r)
        r = fma(r, fma(-x, r, 1.0), r)
        assert abs(Fr(r) - 1 / Fr(x)) <= Fr(0.51) * Fr(float(np.spacing(r)))
        q = a * r
        q = fma(fma(-q, x, a), r, q)
        assert abs(Fr(q) - Fr(a) / Fr(x)) <= Fr(0.51) * Fr(float(np.spacing(abs(q))))
