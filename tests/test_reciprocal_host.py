"""The float32 reciprocal, quotient and square root of the kernels (one Newton-Raphson
step with a fused residual from a hardware approximation), emulated with exact
float64 products: within one ulp of the true value for any approximation that is
itself within two ulps, over the magnitudes the kernels meet."""
import numpy as np
import pytest

F = np.float32


def fma(a, b, c):
    # float32 products are exact in float64; the sum is rounded to float64 and then to
    # float32, which is within 1 + 2^-29 of one float32 rounding
    return (a.astype(np.float64) * b.astype(np.float64) + c.astype(np.float64)).astype(F)


def approx(x, off):
    r = (1.0 / x.astype(np.float64)).astype(F)
    return (r.astype(np.float64) + off * np.spacing(r)).astype(F)


@pytest.mark.parametrize("off", [-2, -1, 0, 1, 2])
def test_reciprocal_quotient_and_root_within_an_ulp(off):
    rng = np.random.default_rng(7)
    x = np.exp(rng.uniform(np.log(1e-6), np.log(1e6), 200000)).astype(F)
    r0 = approx(x, off)
    one = F(1) + np.zeros_like(x)
    r = fma(-r0, fma(x, r0, -one), r0)
    true = 1.0 / x.astype(np.float64)
    assert (np.abs(r - true) <= np.spacing(true.astype(F))).all()
    a = (rng.uniform(-1, 1, x.size) * 10.0 ** rng.uniform(-12, 2, x.size)).astype(F)
    q = (a * r0).astype(F)
    q = fma(fma(-q, x, a), r0, q)
    true = a.astype(np.float64) / x.astype(np.float64)
    assert (np.abs(q - true) <= np.spacing(np.abs(true).astype(F))).all()
    y0 = (1.0 / np.sqrt(x.astype(np.float64))).astype(F)
    y0 = (y0.astype(np.float64) + off * np.spacing(y0)).astype(F)
    s = (x * y0).astype(F)
    s = fma(fma(-s, s, x), (F(0.5) * y0).astype(F), s)
    true = np.sqrt(x.astype(np.float64))
    assert (np.abs(s - true) <= np.spacing(true.astype(F))).all()
