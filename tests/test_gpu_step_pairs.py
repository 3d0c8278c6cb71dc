"""Step calls that take two or three steps per launch (large grids) leave bit for bit
the state of single-step calls: the fused walk repeats the single walk's
operations in order, so nothing but equality is accepted.  The shapes put the
strips' edges everywhere: one strip narrower than a lane pair, a last strip of
one lane, whole strips, wrapped halo columns, short last segments of odd and
even grids, and step counts that mix graphs, whole and part passes and a last
single step."""
import numpy as np
import pytest

from paper_0707_2437_gb300 import workloads

pytestmark = pytest.mark.gpu

# (nx, ny): tiles tall enough that passes of several steps are taken (FP32 strips of
# 112 or 120 columns, 16-bit strips of 240).
SHAPES = {"f32": [(4, 200011), (124, 40003), (1000, 1201), (2048, 1025)],
          "16": [(8, 30011), (248, 20003), (1200, 3607), (2048, 3077)]}


def _state(lbm, kind, nx, ny, calls, lens):
    with lbm.Grid(nx, ny, 0.7, 0.2, kind.replace("-sr", "")) as g:
        if kind.endswith("-sr"):
            g.set_rounding("stochastic")
        if lens:
            g.set_c2_field(workloads.c2_lens(nx, ny, 0.2))
        g.init(*workloads.fourier_modes(nx, ny, amp=1e-2, seed=nx + ny))
        for n in calls:
            g.step(n)
        assert g.t == sum(calls)
        return g.get_state()[0]


@pytest.mark.parametrize("kind,lens", [("f32", False), ("f32", True), ("f16d", False),
                                       ("bf16d", True), ("f16d-sr", False), ("bf16d-sr", False)])
@pytest.mark.parametrize("shape", range(4))
def test_pairs_of_steps_equal_single_steps(lbm, kind, lens, shape):
    nx, ny = SHAPES["f32" if kind == "f32" else "16"][shape]
    single = _state(lbm, kind, nx, ny, [1] * 106, lens)
    pairs = _state(lbm, kind, nx, ny, [2, 100, 1, 3], lens)
    assert np.array_equal(single, pairs)


@pytest.mark.parametrize("nx,ny", [(60, 50021), (1012, 4003)])
def test_three_steps_with_a_c2_field_equal_single_steps(lbm, nx, ny):
    """Grids tall enough for three steps a pass with alpha values in registers: part
    of a strip, and nine whole strips of 112 columns and one of four."""
    single = _state(lbm, "f32", nx, ny, [1] * 14, True)
    assert np.array_equal(single, _state(lbm, "f32", nx, ny, [3, 8, 1, 2], True))


@pytest.mark.parametrize("kind,nx,ny", [
    ("f32", 119, 12001), ("f32", 239, 9001), ("f32", 601, 4001), ("f32", 1001, 1601),
    ("f16d", 238, 9001), ("f16d", 1202, 3001), ("bf16d", 478, 9001),
    ("bf16d-sr", 238, 15001), ("f16d-sr", 1202, 5001)])
def test_passes_at_widths_without_16_byte_lanes(lbm, kind, nx, ny):
    """Rows that start at any word: strips that end inside a lane, wrapped halo columns
    that cross the seam inside one, odd and even row alignments."""
    single = _state(lbm, kind, nx, ny, [1] * 41, False)
    assert np.array_equal(single, _state(lbm, kind, nx, ny, [2, 35, 1, 3], False))
