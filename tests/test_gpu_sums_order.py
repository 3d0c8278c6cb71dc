"""lbm_sums and lbm_sums_noalloc sum in the same order: equal bit for bit, with fewer
reduction blocks than a block has threads, with more, and with the most there are."""
import numpy as np
import pytest

from paper_0707_2437_gb300 import workloads

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("storage", ["f32", "f16d", "bf16d"])
@pytest.mark.parametrize("nx,ny", [(5, 3), (192, 80), (509, 381), (1024, 300)])
def test_totals_agree_bit_for_bit(lbm, storage, nx, ny):
    import torch
    rho, ux, uy = workloads.fourier_modes(nx, ny, amp=1e-2, seed=nx)
    with lbm.Grid(nx, ny, 0.7, 0.2, storage) as g:
        g.init(rho, ux + 1e-3, uy - 2e-3)
        g.step(11)
        want = g.sums()
        dev = torch.from_numpy(g.get_state()[0]).cuda()
        torch.cuda.synchronize()
        got = lbm.sums_noalloc(dev.data_ptr(), nx, ny, nx * ny, storage)
    assert np.array_equal(got, want), (got - want)
