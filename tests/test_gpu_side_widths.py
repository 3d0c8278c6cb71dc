"""Initialisation and moments at widths on both sides of their blocks' column counts, for
one row to more than a block takes: every site's value against numpy.  FP32 values h of
at most a few 1e-1 and weights that sum to one: within 1e-6."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ny", [1, 7, 1025])
@pytest.mark.parametrize("nx", [63, 64, 65, 128, 129, 193, 255, 256, 257, 260, 320, 321, 385, 449,
                                512, 513, 2049])
def test_fields_in_and_out(lbm, nx, ny):
    import torch
    rng = np.random.default_rng(nx * ny)
    f = [rng.uniform(0.95, 1.05, (ny, nx))] + [rng.uniform(-0.05, 0.05, (ny, nx)) for _ in range(2)]
    with lbm.Grid(nx, ny, 0.8, 0.2) as g:
        g.init(*[torch.from_numpy(a).cuda() for a in f])
        out = [torch.full((ny, nx), np.nan, dtype=torch.float64, device="cuda") for _ in range(3)]
        g.moments(out)
        for a, b in zip(f, out):
            assert np.abs(a - b.cpu().numpy()).max() < 1e-6
