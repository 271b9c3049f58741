"""The largest gradient of lbm_interface_width where the squares of the gradients lie below
the normal range of float32: the value of the returned density all the same (1e-14, the same
float64 differences on both sides)."""
import numpy as np
import pytest

import oracle as O
from cases import case, lbm_params
from paper_2201_12404_gb300 import lbm

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("D", [2, 3])
def test_gradients_whose_squares_underflow_float32(D):
    c = case(D, 40, 12, 12, precision=lbm.LBM_FP64)
    sh = (c["nz"], c["ny"], c["nx"])
    rho = np.full(sh, 1e-10)
    z, y = sh[0] // 2, sh[1] // 2
    for ax in range(D):  # one node with a difference along every axis, one with a larger along x alone
        at = [z, y, 8]
        at[2 - ax] += 1
        rho[tuple(at)] += 2.2e-23
    rho[z, y, 21] += 2.8e-23
    f = O.weights(D).reshape((-1, 1, 1, 1)) * rho
    with lbm.Domain(lbm_params(c)) as dom:
        dom.lbm_write_populations(f)
        r, _ = dom.lbm_read_macroscopic()
        grad = dom.lbm_interface_width()[1]
    g2 = sum((0.5 * (np.roll(r, -1, axis) - np.roll(r, 1, axis))) ** 2 for axis in range(3 - D, 3))
    assert grad == pytest.approx(np.sqrt(g2.max()), rel=1e-14, abs=0)
