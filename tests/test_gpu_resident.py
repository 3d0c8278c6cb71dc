"""Calls that run resident (one launch, the grid's tiles in shared memory) leave
bit for bit the state the step kernel leaves: the same operations in the same
order, so nothing but equality is accepted.  The sizes are single tiles, cuts in
one and in both directions, odd widths and heights, tiles whose halo is the whole
neighbour, and the largest that run this way; the step counts end before, at and
after exchanges of tile edges, with an even and an odd number of them."""
import numpy as np
import pytest

from paper_0707_2437_gb300 import workloads

pytestmark = pytest.mark.gpu

SIZES = [(1, 1), (5, 1), (1, 9), (16, 3), (37, 23), (400, 4), (3, 700), (8192, 4), (64, 64),
         (130, 9), (250, 252), (509, 381), (600, 590)]


def _state(lbm, nx, ny, kind, option, calls, resident):
    with lbm.Grid(nx, ny, 0.7, 0.2, kind.replace("-sr", "")) as g:
        if kind.endswith("-sr"):
            g.set_rounding("stochastic")
        if option == "field":
            g.set_c2_field(workloads.c2_lens(nx, ny, 0.2))
        if option == "drive":
            g.set_drive(1e-3, 40.0)
        if not resident:
            g.set_persistent(False)
        g.init(*workloads.fourier_modes(nx, ny, amp=1e-2, seed=nx + ny))
        for n in calls:
            g.step(n)
        g.sync()
        assert g.t == sum(calls)
        return g.get_state()[0]


@pytest.mark.parametrize("nx,ny", SIZES)
@pytest.mark.parametrize("kind,option", [("f32", ""), ("f32", "field"), ("f32", "drive"),
                                         ("f16d", ""), ("bf16d", "field"), ("f16d-sr", ""),
                                         ("bf16d-sr", "drive")])
def test_resident_steps_equal_step_kernel(lbm, nx, ny, kind, option):
    if option == "drive" and nx < 4:
        pytest.skip("a driven channel needs nx >= 4")
    calls = [4, 1, 17, 150, 5, 64]  # (the drive's values come in chunks of 128)
    a = _state(lbm, nx, ny, kind, option, calls, True)
    b = _state(lbm, nx, ny, kind, option, calls, False)
    assert np.array_equal(a, b)


def test_resident_grids_on_several_streams(lbm):
    """Grids stepped resident on streams of their own, interleaved, reach their
    solo states."""
    sizes = [(256, 256), (400, 4), (200, 300), (64, 64)]
    streams = [lbm.new_stream() for _ in sizes]
    grids = []
    for (nx, ny), s in zip(sizes, streams):
        g = lbm.Grid(nx, ny, 0.8, 0.2, "f32", stream=s)
        g.init(*workloads.fourier_modes(nx, ny, amp=1e-3, seed=nx))
        grids.append(g)
    for _ in range(3):
        for g in grids:
            g.step(40)
    for (nx, ny), g in zip(sizes, grids):
        got = g.get_state()[0]
        g.close()
        with lbm.Grid(nx, ny, 0.8, 0.2, "f32") as h:
            h.set_persistent(False)
            h.init(*workloads.fourier_modes(nx, ny, amp=1e-3, seed=nx))
            h.step(120)
            assert np.array_equal(h.get_state()[0], got)
