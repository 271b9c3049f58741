"""psi inside the interface band on the float32 path, from two cubics in the density
carried as pairs of float32 and rounded once, emulated with numpy."""
import numpy as np
import pytest

F, D = np.float32, np.float64


def fma(a, b, c):
    # float32 products are exact in float64; one rounding to float64 and one to float32
    return (a.astype(D) * b.astype(D) + c.astype(D)).astype(F)


def split(c):
    h = F(c)
    return h, F(c - D(h))


def cubic(c, x):
    h, l = (v + F(0) * x for v in split(c[3]))
    for k in (2, 1, 0):
        ch, cl = split(c[k])
        p = h * x
        ep = fma(l, x, fma(h, x, -p))
        h = p + ch
        b = h - p
        l = ((p - (h - b)) + (ch - b)) + (ep + cl)
    s = h + l
    return s, l - (s - h)


def psi_pairs(num, den, rho, off):
    nh, nl = cubic(num, rho)
    mh, ml = cubic(den, rho)
    r = (1.0 / mh.astype(D)).astype(F)
    r = (r.astype(D) + off * np.spacing(r)).astype(F)
    q = nh * r
    qt = fma(-q, ml, fma(-q, mh, nh) + nl) * r
    v = q * rho
    vt = fma(qt, rho, fma(q, rho, -v))
    sign = np.where(v < 0, F(-1), F(1))
    v, vt = sign * v, sign * vt
    y = (1.0 / np.sqrt(v.astype(D))).astype(F)
    y = (y.astype(D) + off * np.spacing(y)).astype(F)
    s = v * y
    return np.where(v < F(1.2e-38), F(0), fma(fma(-s, s, v) + vt, F(0.5) * y, s))


@pytest.mark.parametrize("off", [-2, 0, 2])
@pytest.mark.parametrize("T", [0.55, 0.75, 0.97])
@pytest.mark.parametrize("a", [0.003, 3.0 / 49.0, 0.5])
def test_psi_by_pairs_is_rounded_once(a, T, off):
    """b = 2/21, omega = 0.344 at T T_c; with a = 0.5, P = rho/3 has roots.
    Half an ulp from the one rounding and 2^-20 of it from the quotient's and the root's
    second terms, and near a root the 2^-44 of the cubic's terms."""
    b, w = 2.0 / 21.0, 0.344
    RT = 0.0778 / 0.45724 * a / b * T
    m = 0.37464 + 1.54226 * w - 0.26992 * w * w
    aal = a * (1 + m * (1 - np.sqrt(T))) ** 2
    num = [3 * RT - 1, (6 * RT - 1) * b - 3 * aal, ((3 - 3 * RT) * b + 3 * aal) * b, -b ** 3]
    den = [3.0, 3 * b, -9 * b * b, 3 * b ** 3]
    rng = np.random.default_rng(3)
    rho = rng.uniform(0.02, 9.0, 200000).astype(F)
    for root in np.roots(num[::-1]):
        if abs(root.imag) < 1e-12 and 0.02 < root.real < 9.0:
            near = F(root.real) + np.arange(-50, 51) * np.spacing(F(root.real))
            rho = np.concatenate([rho, near.astype(F)])
    L = np.longdouble
    x, one = rho.astype(L), L(1)
    t = L(b) * x
    terms = [L(RT) * x / (one - t), L(aal) * x * x / (one + 2 * t - t * t), x / 3]
    v = np.abs(terms[0] - terms[1] - terms[2])
    exact = np.sqrt(v)
    got = psi_pairs(num, den, rho, off)
    size = sum(abs(L(c)) * x ** k for k, c in enumerate(num)) * x / (3 * (one - t) * (one + 2 * t - t * t))
    bound = 0.5 * (1 + 2.0 ** -12) * np.spacing(exact.astype(F)).astype(L) + 2.0 ** -44 * size / (2 * np.maximum(exact, 1e-30))
    ok = (np.abs(got - exact) <= bound) | (v < 2.0 ** -43 * size)
    assert ok.all(), (rho[~ok][:5], got[~ok][:5], exact[~ok][:5])
