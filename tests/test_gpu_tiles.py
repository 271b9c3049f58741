"""The tiled kernels where lanes of a tile lie outside the domain, against the oracle:
passes 1 and 2 of 3-D domains that tiles cover with less than 8% to spare (others take
consecutive nodes of a layer), and the large tile of pass 1b (32x4x6 nodes in 3-D, 64x16 in
2-D), which only large domains take.  Tolerances per step as in test_gpu_parity and
test_gpu_fp16dev."""
import numpy as np
import pytest

import oracle as O
from cases import case, drop_state, lbm_params, oracle_params, rel_err
from paper_2201_12404_gb300 import lbm
from test_gpu_fp16dev import TOL_STEP, host_codec
from test_gpu_parity import TOL, as_storage, run_both

pytestmark = pytest.mark.gpu

WALLS = [False, (0,), (1,), (0, 1, 2)]


def tiles(shape, tile):
    return np.prod([-(-n // t) for n, t in zip(shape, tile)])


@pytest.mark.parametrize("walls", WALLS)
@pytest.mark.parametrize("shape", [(31, 16, 5), (31, 32, 6), (62, 31, 7), (95, 33, 9)])
@pytest.mark.parametrize("precision", [lbm.LBM_FP64, lbm.LBM_FP32, lbm.LBM_FP16DEV], ids=["fp64", "fp32", "fp16dev"])
def test_partly_filled_tiles_of_passes_1_and_2(shape, walls, precision):
    nodes = shape[0] * shape[1]
    assert nodes < tiles(shape[:2], (32, 2)) * 64 <= 1.08 * nodes
    c = case(3, *shape, walls=walls, precision=precision)
    f0 = drop_state(c)
    if precision == lbm.LBM_FP16DEV:
        with lbm.Domain(lbm_params(c)) as dom:
            dom.lbm_write_populations(f0)
            dom.lbm_step(2)
            fg = dom.lbm_read_populations()
        fo, _ = O.run(oracle_params(c), host_codec(f0, c), 2)
        assert rel_err(fg, fo, 3).max() <= 2 * TOL_STEP
    else:
        fg, fo = run_both(c, as_storage(f0, precision), 3)
        assert rel_err(fg, fo, 3).max() <= 4 * TOL[precision]


@pytest.mark.parametrize("walls", [False, (0,), (1,), (0, 1)])
@pytest.mark.parametrize("precision", [lbm.LBM_FP64, lbm.LBM_FP32], ids=["fp64", "fp32"])
def test_large_tile_of_pass_1b_2d(walls, precision):
    shape = (650, 701)
    assert tiles(shape, (64, 16)) >= 3 * 152
    c = case(2, *shape, walls=walls, precision=precision)
    fg, fo = run_both(c, as_storage(drop_state(c), precision), 3)
    assert rel_err(fg, fo, 2).max() <= 4 * TOL[precision]


@pytest.mark.parametrize("walls", WALLS)
def test_large_tile_of_pass_1b_3d_float64(walls):
    shape = (67, 41, 163)
    assert tiles(shape, (32, 4, 6)) >= 6 * 152
    c = case(3, *shape, walls=walls)
    fg, fo = run_both(c, drop_state(c), 2)
    assert rel_err(fg, fo, 3).max() <= 4 * TOL[lbm.LBM_FP64]


@pytest.mark.parametrize("walls", WALLS)
def test_large_tile_of_pass_1b_3d_float32(walls):
    """A state of period 61 along z: away from walls on z the domain of one period gives every
    period of the run, next to them the domain of two periods between such walls."""
    nx, ny, period, count, steps = 33, 5, 61, 598, 2
    assert tiles((nx, ny, period * count), (32, 4, 6)) >= 160 * 152
    one = case(3, nx, ny, period, walls=tuple(a for a in walls or () if a < 2), precision=lbm.LBM_FP32)
    f0 = as_storage(drop_state(one), lbm.LBM_FP32)
    inner, _ = O.run(oracle_params(one), f0, steps)
    lowest = highest = inner
    if walls and 2 in walls:
        ends, _ = O.run(oracle_params(case(3, nx, ny, 2 * period, walls=walls)), np.tile(f0, (1, 2, 1, 1)), steps)
        lowest, highest = ends[:, :period], ends[:, period:]
    with lbm.Domain(lbm_params(case(3, nx, ny, period * count, walls=walls, precision=lbm.LBM_FP32))) as dom:
        dom.lbm_write_populations(np.tile(f0, (1, count, 1, 1)))
        dom.lbm_step(steps)
        dom.lbm_synchronize()
        for k, fo in ((0, lowest), (1, inner), (2, inner), (301, inner), (count - 2, inner), (count - 1, highest)):
            fg = dom.lbm_read_populations_window((0, 0, period * k), (nx, ny, period))
            assert rel_err(fg, fo, 3).max() <= 4 * TOL[lbm.LBM_FP32], k
