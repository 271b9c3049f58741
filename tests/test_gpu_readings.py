"""The readings reduced on the GPU against the fields the library returns, at sizes
around the edges of the reduction tiles (32 x 8 nodes) and beyond one tile per block.

Tolerances: the totals are float64 sums of the same populations in another order, at
most 10 roundings deep per term on either side (1e-13 of the sum of magnitudes); the
largest speed and gradient take the same float64 values (1e-14)."""
import numpy as np
import pytest

import oracle as O
from cases import case, lbm_params
from paper_2201_12404_gb300 import inputs as I
from paper_2201_12404_gb300 import lbm

pytestmark = pytest.mark.gpu

SIZES = {"2d_tile": dict(D=2, nx=32, ny=8), "2d_ragged": dict(D=2, nx=33, ny=9, walls=True),
         "2d_many_tiles": dict(D=2, nx=1030, ny=515), "3d_min": dict(D=3, nx=5, ny=5, nz=5),
         "3d_ragged": dict(D=3, nx=65, ny=17, nz=9, walls=True)}


@pytest.mark.parametrize("precision", [lbm.LBM_FP64, lbm.LBM_FP32, lbm.LBM_FP16DEV], ids=["fp64", "fp32", "fp16dev"])
@pytest.mark.parametrize("name", list(SIZES))
def test_readings_match_the_returned_fields(name, precision):
    c = case(**SIZES[name], Tr=0.8, precision=precision)
    D, sh = c["D"], (c["nz"], c["ny"], c["nx"])
    rho = I.drop(sh, (c["nx"] / 2, c["ny"] / 2, c["nz"] / 2), 0.3 * min(s for s in sh if s > 1), c["rho_l"], c["rho_v"], 4.0, D=D)
    u = I.rng(5).uniform(-0.02, 0.02, (D,) + sh)
    with lbm.Domain(lbm_params(c)) as dom:
        dom.lbm_init_fields(rho, u)
        dom.lbm_step(1)  # odd parity: the gather crosses nodes
        diag = dom.lbm_read_diag()
        speed, (width, grad) = dom.lbm_max_speed(), dom.lbm_interface_width()
        f = dom.lbm_read_populations()
        r, v = dom.lbm_read_macroscopic()
    vel = O.velocities(D)
    node_rho = f.sum(axis=0)
    mom = [np.tensordot(vel[:, a].astype(float), f, axes=1) for a in range(3)]
    total = np.abs(f).sum()
    assert abs(diag["mass"] - node_rho.sum()) <= 1e-13 * total
    for a in range(D):
        assert abs(diag["momentum"][a] - mom[a].sum()) <= 1e-13 * total
    bare = np.sqrt(sum(m * m for m in mom)) / node_rho
    assert diag["max_u"] == pytest.approx(bare.max(), rel=1e-12)
    assert speed == pytest.approx(np.sqrt((v ** 2).sum(axis=0)).max(), rel=1e-14)
    g2 = np.zeros(sh)
    for ax, axis in ((0, 2), (1, 1), (2, 0)):
        if ax >= D:
            continue
        mode = "symmetric" if c["bc"][2 * ax] else "wrap"
        p = np.pad(r, [(1, 1) if k == axis else (0, 0) for k in range(3)], mode=mode)
        lo, hi = [slice(None)] * 3, [slice(None)] * 3
        lo[axis], hi[axis] = slice(0, -2), slice(2, None)
        g2 += (0.5 * (p[tuple(hi)] - p[tuple(lo)])) ** 2
    assert grad == pytest.approx(np.sqrt(g2.max()), rel=1e-14)
    assert width == pytest.approx((c["rho_l"] - c["rho_v"]) / grad, rel=1e-14)
