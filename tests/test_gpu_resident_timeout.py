"""A wait inside a resident launch that runs out: with a limit of zero a block gives up
when a neighbour's counter is not there at the first look, which some of the 152 blocks
meet in 200 exchanges (limits of 1 us do not run out: the waits are shorter).  The launch
ends, the host reads LBM_ETIMEOUT once, and the grid steps on correctly after a new
start."""
import numpy as np
import pytest

from paper_0707_2437_gb300 import workloads

pytestmark = pytest.mark.gpu


def test_bad_arguments(lbm):
    lib = lbm.load()
    assert lib.lbm_set_timeout_us(None, 1000) == -1
    with lbm.Grid(16, 16, 0.8, 0.2) as g:
        assert lib.lbm_set_timeout_us(g.h, -1) == -1


@pytest.mark.parametrize("read", ["sync", "sums", "moments", "get_state"])
def test_resident_timeout_reports_status(lbm, read):
    nx, ny = 256, 256
    fields = workloads.fourier_modes(nx, ny, amp=1e-2, seed=7)
    with lbm.Grid(nx, ny, 0.8, 0.2) as g:
        g.init(*fields)
        assert g.step_form(600) == ("resident", 600)
        g.set_timeout_us(0)
        g.step(600)
        with pytest.raises(lbm.LbmError) as ei:
            getattr(g, read)()
        assert ei.value.status == lbm.LBM_ETIMEOUT
        g.sync()  # reported once
        g.set_timeout_us(1_000_000)
        g.init(*fields)
        g.step(90)
        g.sync()
        assert g.t == 90
        state = g.get_state()[0]
        g.set_persistent(False)
        g.init(*fields)
        g.step(90)
        assert np.array_equal(g.get_state()[0], state)
