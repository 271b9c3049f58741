"""Mass of a fluid at rest in float32: over 50 steps of a uniform domain it stays within 8
units in the last place of the density (8 2^-24).  A rounding that falls the same way at every
node and step would take some units a step."""
import numpy as np
import pytest

from cases import case, lbm_params, shape
from paper_2201_12404_gb300 import lbm

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("phase", ["rho_l", "rho_v"])
@pytest.mark.parametrize("Tr", [0.6, 0.75, 0.8, 0.9])
@pytest.mark.parametrize("D", [2, 3])
def test_uniform_domain_keeps_its_mass(D, Tr, phase):
    dims = dict(nx=64, ny=48) if D == 2 else dict(nx=32, ny=24, nz=16)
    c = case(D, **dims, Tr=Tr, precision=lbm.LBM_FP32)
    with lbm.Domain(lbm_params(c)) as dom:
        dom.lbm_init_fields(np.full(shape(c), c[phase]), np.zeros((D,) + shape(c)))
        start = dom.lbm_read_diag()["mass"]
        dom.lbm_step(50)
        end = dom.lbm_read_diag()["mass"]
    assert abs(end - start) <= 8 * 2.0 ** -24 * start
