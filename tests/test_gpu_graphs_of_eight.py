"""Calls of lbm_step with eight steps and more left replay graphs of eight steps: bit for bit
the state and the gamma record of a domain stepped kernel by kernel (timing on), from both
parities, with and without rests of two steps and of one, and with the gamma record switched
on and off between calls."""
import numpy as np
import pytest

from cases import case, drop_state, lbm_params
from paper_2201_12404_gb300 import lbm

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("D,precision", [(3, lbm.LBM_FP32), (2, lbm.LBM_FP32), (3, lbm.LBM_FP64), (2, lbm.LBM_FP64),
                                         (3, lbm.LBM_FP16DEV), (2, lbm.LBM_FP16DEV)])
def test_eight_step_graphs_equal_kernel_by_kernel_steps(D, precision):
    dims = dict(nx=40, ny=22, nz=13) if D == 3 else dict(nx=70, ny=37)
    c = case(D, **dims, precision=precision, walls=True)
    f0 = drop_state(c, perturb=0.002)
    with lbm.Domain(lbm_params(c)) as plain, lbm.Domain(lbm_params(c)) as graphed:
        for d in (plain, graphed):
            d.lbm_write_populations(f0)
        plain.lbm_set_timing(True)
        n0, steps = graphed.lbm_launch_count(), 0
        # (steps, gamma record): 2 + 8 + 1 ends at odd parity, where 8, then 16 + 2 + 1, begin
        for n, gamma in ((11, False), (8, False), (19, False), (17, True), (8, True), (10, False), (9, True)):
            for d in (plain, graphed):
                d.lbm_record_gamma(gamma)
                d.lbm_step(n)
            steps += n
            assert np.array_equal(plain.lbm_read_populations(), graphed.lbm_read_populations()), steps
            if gamma:
                a, b = (d.lbm_read_diag(with_gamma=True)["gamma"] for d in (plain, graphed))
                assert np.array_equal(a, b), steps
        assert np.isfinite(graphed.lbm_read_populations()).all()
        assert graphed.lbm_launch_count() - n0 >= 3 * steps
