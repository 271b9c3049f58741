"""A reading whose kernel may give up a bounded wait reports it: with bit 1 of the domain's
error word set, as such a kernel leaves it, lbm_max_speed returns LBM_ERR_TIMEOUT in place of
a maximum over the tiles that arrived."""
import ctypes

import pytest

from cases import case, drop_state, lbm_params
from paper_2201_12404_gb300 import lbm

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("reading", ["lbm_max_speed", "lbm_interface_width"])
def test_a_wait_that_gave_up_is_reported(reading):
    c = case(2, 70, 37, precision=lbm.LBM_FP32)
    held = {}

    def alloc(nbytes, ctx):
        t = torch.zeros(int(nbytes), dtype=torch.uint8, device="cuda")
        held[t.data_ptr()] = t
        return t.data_ptr()

    p = lbm_params(c)
    p.dev_alloc, p.dev_free = lbm.DEV_ALLOC(alloc), lbm.DEV_FREE(lambda ptr, ctx: held.pop(int(ptr), None))
    with lbm.Domain(p) as dom:
        dom.lbm_write_populations(drop_state(c))
        dom.lbm_step(1)
        dom.lbm_synchronize()
        getattr(dom, reading)()
        # the error word is the domain's smallest buffer
        word = min(held.values(), key=lambda t: t.numel())
        assert word.numel() == ctypes.sizeof(ctypes.c_uint) + 2 * ctypes.sizeof(ctypes.c_ulonglong)
        word[0] = 2
        torch.cuda.synchronize()
        with pytest.raises(lbm.LBMError) as e:
            getattr(dom, reading)()
        assert e.value.status == lbm.LBM_ERR_TIMEOUT
