"""lbm_mode on thin grids, against the same sums in numpy from the stored distributions:
grids of a few rows with more columns than one round of blocks takes (their blocks are
wider), narrow ones (whose blocks take fewer rows), and the edges between.

Bound.  Both sides add the same N terms v cos(phase) in FP64 in different orders and
scale by 2/N: each sum errs by at most about the length of its longest chain (1024 terms
here, in numpy's pairwise sums fewer) times 2^-53 times the mean of |v|, the phase
factors by a few 2^-53: 2e-13 of the largest |v|, with a factor of ten to spare below."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

EX = (0, 1, 0, -1, 0, 1, -1, -1, 1)
EY = (0, 0, 1, 0, -1, 1, 1, -1, -1)
W = (4 / 9,) + (1 / 9,) * 4 + (1 / 36,) * 4


@pytest.mark.parametrize("nx,ny", [(40000, 2), (70000, 1), (140000, 1), (270000, 1), (33000, 4),
                                   (33000, 5), (32768, 3), (4, 400), (1, 700), (9, 65), (31, 64),
                                   (3, 20000)])
def test_modes_of_thin_grids(lbm, nx, ny):
    rng = np.random.default_rng(nx + ny)
    rho = 1.0 + 1e-2 * rng.standard_normal((ny, nx))
    ux, uy = (1e-2 * rng.standard_normal((ny, nx)) for _ in range(2))
    with lbm.Grid(nx, ny, 0.8, 0.2) as g:
        g.init(rho, ux, uy)
        h = g.get_state()[0].view(np.float32).reshape(9, ny, nx).astype(np.float64)
        # plane i holds at x the value that streams to x + e_i
        f = [W[i] * np.roll(h[i], (EY[i], EX[i]), (0, 1)) for i in range(9)]
        dr = sum(f)
        fields = {"rho": dr, "ux": sum(EX[i] * f[i] for i in range(9)) / (1.0 + dr),
                  "uy": sum(EY[i] * f[i] for i in range(9)) / (1.0 + dr)}
        for kx, ky in ((1, 0), (0, 1), (3, 2), (-2, 5)):
            # phases reduced exactly before scaling
            px = 2.0 * np.pi * ((kx * np.arange(nx)) % nx / nx)[None, :]
            py = 2.0 * np.pi * ((ky * np.arange(ny)) % ny / ny)[:, None]
            for name, v in fields.items():
                want = 2.0 / (nx * ny) * np.array([(v * np.cos(px + py)).sum(),
                                                   (v * np.sin(px + py)).sum()])
                got = g.mode(name, kx, ky)
                assert np.abs(got - want).max() <= 2e-12 * np.abs(v).max(), (name, kx, ky)
