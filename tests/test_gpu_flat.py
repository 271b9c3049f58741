"""Both mappings of passes 1 and 2 in 3-D, tiles (rows of a multiple of 32 nodes) and
consecutive nodes of a layer (the other sizes), against the oracle over both parities."""
import pytest

from cases import case, drop_state, rel_err
from paper_2201_12404_gb300 import lbm
from test_gpu_parity import TOL, as_storage, run_both

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("walls", [False, (0,), (1,), (2,), (0, 1, 2)])
@pytest.mark.parametrize("shape", [(5, 5, 5), (16, 8, 5), (33, 6, 5), (65, 5, 6), (129, 5, 5), (32, 6, 5), (64, 8, 5)])
@pytest.mark.parametrize("precision", [lbm.LBM_FP64, lbm.LBM_FP32], ids=["fp64", "fp32"])
def test_mappings_match_oracle(shape, walls, precision):
    c = case(3, *shape, walls=walls, precision=precision)
    f0 = as_storage(drop_state(c), precision)
    fg, fo = run_both(c, f0, 2)
    assert rel_err(fg, fo, 3).max() <= 4 * TOL[precision]
