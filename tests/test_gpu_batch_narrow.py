"""FP32 batches whose grids have one strip more in passes of two steps (strips of 120
columns) than in single steps (128): less than a wave of tiles steps singly, more takes
passes.  The number of tiles tells which; states are those of grids stepped alone, bit
for bit."""
import numpy as np
import pytest

from paper_0707_2437_gb300 import workloads

pytestmark = pytest.mark.gpu


def _grid(lbm, nx, ny, k, lens):
    g = lbm.Grid(nx, ny, 0.6 + 0.01 * k, 0.2)
    if lens:
        g.set_c2_field(workloads.c2_lens(nx, ny, 0.2))
    g.init(*workloads.fourier_modes(nx, ny, amp=1e-2, seed=k))
    return g


@pytest.mark.parametrize("schedule", ["lockstep", "flow"])
@pytest.mark.parametrize("lens", [False, True])
@pytest.mark.parametrize("count,nx,ny,single", [(64, 124, 256, False), (128, 124, 64, True),
                                                (64, 116, 128, False), (9, 128, 4096, False)])
def test_narrow_batches(lbm, schedule, lens, count, nx, ny, single):
    grids = [_grid(lbm, nx, ny, k, lens) for k in range(count)]
    b = lbm.Batch(grids)
    b.set_schedule(schedule)
    # (single steps: tiles of four rows in one strip)
    tiles = b.get_config()["tiles"]
    assert (tiles == count * ny // 4) == single, tiles
    b.step(7, [1 + k % 7 for k in range(count)])
    b.step(2)
    assert b.sync() == 0
    got = {k: grids[k].get_state()[0] for k in (0, 1, 5, count - 1)}
    b.close()
    for g in grids:
        g.close()
    for k, state in got.items():
        with _grid(lbm, nx, ny, k, lens) as h:
            for _ in range(3 + k % 7):
                h.step(1)
            assert np.array_equal(h.get_state()[0], state)
