"""Blocks of the batch kernel whose consecutive share of the tiles crosses jobs: more jobs
than blocks, of three sizes, each bit for bit as the domain stepped alone."""
import numpy as np
import pytest

from cases import case, drop_state, lbm_params
from paper_2201_12404_gb300 import lbm

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("count", [1, 2, 1201])
@pytest.mark.parametrize("precision", [lbm.LBM_FP32, lbm.LBM_FP64], ids=["fp32", "fp64"])
def test_shares_that_cross_jobs_equal_single_domains(count, precision):
    kinds = [case(2, nx, ny, precision=precision) for nx, ny in ((9, 5), (70, 11), (33, 6))]
    start = [drop_state(c) for c in kinds]
    ref = []
    for c, f0 in zip(kinds, start):
        with lbm.Domain(lbm_params(c)) as d:
            d.lbm_write_populations(f0)
            d.lbm_step(3)
            ref.append(d.lbm_read_populations())
    doms = []
    for k in range(count):
        d = lbm.Domain(lbm_params(kinds[k % 3]))
        d.lbm_write_populations(start[k % 3])
        doms.append(d)
    with lbm.Batch(doms) as b:
        b.lbm_batch_step(3)
        b.lbm_batch_synchronize()
    for k in list(range(min(count, 30))) + list(range(max(0, count - 30), count)) + list(range(0, count, 37)):
        assert np.array_equal(doms[k].lbm_read_populations(), ref[k % 3])
    for d in doms:
        d.close()
