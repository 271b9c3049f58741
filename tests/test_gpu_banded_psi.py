"""The default EOS mode of the float32 path: pairs of float32 inside the interface band, and
float64 there where the parameters are out of the pairs' range (a = 1e-9: P nearly 0)."""
import pytest

from cases import case, drop_state, rel_err
from paper_2201_12404_gb300 import lbm
from test_gpu_parity import TOL, as_storage, run_both

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("a", [0.003, 0.5, 1e-9])
@pytest.mark.parametrize("D", [2, 3])
def test_band_matches_oracle(D, a):
    c = case(D, 35, 24, 9 if D == 3 else 1, a=a, Tr=0.6, rho_l=1.0, rho_v=0.2, kappa=0.001, precision=lbm.LBM_FP32)
    f0 = as_storage(drop_state(c, perturb=0.002), lbm.LBM_FP32)
    fg, fo = run_both(c, f0, 1)
    assert rel_err(fg, fo, D).max() <= TOL[lbm.LBM_FP32]
