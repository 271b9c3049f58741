"""The largest speed of lbm_read_diag where all speeds are small against the rounding of
a momentum formed in float32, or the density is small against its populations: the value
of the populations in float64 all the same, and the same value on every call.

Tolerance: both sides form every node's speed in float64 from the same populations,
sums of 27 terms of magnitude S = sum |f| in different orders: 30 S 2^-53 on a momentum
or a density, relative to the momentum and to the density of the fastest node."""
import numpy as np
import pytest

import oracle as O
from cases import case, lbm_params
from paper_2201_12404_gb300 import lbm

pytestmark = pytest.mark.gpu

SHAPES = {2: dict(nx=300, ny=203), 3: dict(nx=97, ny=45, nz=33)}


def speeds(f, D):
    vel = O.velocities(D).astype(float)
    rho, size = f.sum(axis=0), np.abs(f).sum(axis=0)
    j = np.sqrt(sum(np.tensordot(vel[:, a], f, axes=1) ** 2 for a in range(D)))
    return j / rho, 30 * 2.0 ** -53 * size * (1 / np.maximum(j, 1e-300) + 1 / np.abs(rho))


def state(c, kind):
    D, sh = c["D"], (c["nz"], c["ny"], c["nx"])
    r = np.random.default_rng(4)
    w = O.weights(D).reshape((-1, 1, 1, 1))
    vel = O.velocities(D).astype(float)
    rho = np.full(sh, 5.0) + r.uniform(-1e-3, 1e-3, sh)
    if kind == "cancelling":  # the rest population takes back what the others carry
        f = w * rho * (1 + 1e-3 * r.uniform(-1, 1, (len(w),) + sh))
        rest = len(w) // 2
        f[rest] = -(f.sum(axis=0) - f[rest]) + 1e-5
        return f
    z, y, x = np.meshgrid(*(np.arange(n) for n in sh), indexing="ij")
    a, b = 2 * np.pi * x / sh[2], 2 * np.pi * y / sh[1]
    u = [kind * np.sin(a) * np.cos(b), -kind * np.cos(a) * np.sin(b), 0.3 * kind * np.cos(a + b)]
    return w * rho * (1 + 3 * sum(vel[:, k].reshape((-1, 1, 1, 1)) * u[k] for k in range(D)))


@pytest.mark.parametrize("kind", [1e-8, 1e-7, 1e-6, 1e-5, 1e-4, 1e-3, "cancelling"])
@pytest.mark.parametrize("D", [2, 3])
def test_largest_speed_is_that_of_the_populations(D, kind):
    c = case(D, **SHAPES[D], precision=lbm.LBM_FP32)
    f = state(c, kind).astype(np.float32).astype(np.float64)
    with lbm.Domain(lbm_params(c)) as dom:
        dom.lbm_write_populations(f)
        got = [dom.lbm_read_diag()["max_u"] for _ in range(5)]
    u, tol = speeds(f, D)
    top = np.unravel_index(u.argmax(), u.shape)
    assert len(set(got)) == 1, got
    assert abs(got[0] - u[top]) <= (tol[top] + 1e-15) * u[top], (got[0], u[top])
