"""Batches whose passes take two or three steps (the fused walk) leave every grid bit
for bit in the state single steps leave it in, in both schedules: odd and even
step limits, limits that end early, tile heights from one row up (the flow
schedule uses at least four, the reach of a pass), strips of one lane, one whole
strip and a last strip of one lane (120 columns in FP32, 240 in 16 bits)."""
import numpy as np
import pytest

from paper_0707_2437_gb300 import workloads

pytestmark = pytest.mark.gpu

SIZES = [(8, 3), (16, 1), (120, 4), (124, 7), (240, 33), (248, 5), (256, 100), (488, 20)]


def _grid(lbm, kind, lens, k):
    nx, ny = SIZES[k]
    if kind == "mixed":
        kind = "f16d" if k % 2 else "f32"
    if kind == "f32" and nx == 248:
        nx = 244
    g = lbm.Grid(nx, ny, 0.6 + 0.05 * k, 0.1 + 0.04 * k, kind.replace("-sr", ""))
    if kind.endswith("-sr"):
        g.set_rounding("stochastic")
    if lens:
        g.set_c2_field(workloads.c2_lens(nx, ny, 0.2))
    g.init(*workloads.fourier_modes(nx, ny, amp=1e-2, seed=k))
    return g


@pytest.mark.parametrize("schedule", ["lockstep", "flow"])
@pytest.mark.parametrize("rows", [None, 1, 5])
@pytest.mark.parametrize("kind,lens", [("f32", False), ("f32", True), ("f16d", False),
                                       ("bf16d", True), ("f16d-sr", False), ("mixed", False)])
def test_pairs_in_batches_equal_single_steps(lbm, kind, lens, rows, schedule):
    limits = [1 + (7 * k) % 12 for k in range(len(SIZES))]
    grids = [_grid(lbm, kind, lens, k) for k in range(len(SIZES))]
    b = lbm.Batch(grids)
    b.set_schedule(schedule)
    if rows:
        b.set_config(rows, 0)
    b.step(12, limits)
    b.step(3)
    b.step(1, [k % 2 for k in range(len(SIZES))])
    assert b.sync() == 0
    got = [(g.t, g.get_state()[0]) for g in grids]
    b.close()
    for g in grids:
        g.close()
    for k, (t, state) in enumerate(got):
        with _grid(lbm, kind, lens, k) as h:
            for _ in range(limits[k] + 3 + k % 2):
                h.step(1)
            assert h.t == t
            assert np.array_equal(h.get_state()[0], state), SIZES[k]


def test_tall_tiles_in_a_batch_equal_single_steps(lbm):
    """Grids tall enough for FP32's passes of three steps in lockstep (tiles over 64
    rows on every resident warp), with limits that leave one and two steps."""
    sizes, limits = [(64, 100003), (124, 20001)], [10, 8]
    fields = [workloads.fourier_modes(nx, ny, amp=1e-2, seed=nx) for nx, ny in sizes]
    grids = []
    for (nx, ny), f in zip(sizes, fields):
        g = lbm.Grid(nx, ny, 0.7, 0.2)
        g.init(*f)
        grids.append(g)
    b = lbm.Batch(grids)
    assert b.get_config()["rows"] > 64
    b.step(10, limits)
    b.step(3)
    assert b.sync() == 0
    got = [g.get_state()[0] for g in grids]
    b.close()
    for g in grids:
        g.close()
    for (nx, ny), f, n, state in zip(sizes, fields, limits, got):
        with lbm.Grid(nx, ny, 0.7, 0.2) as h:
            h.init(*f)
            for _ in range(n + 3):
                h.step(1)
            assert np.array_equal(h.get_state()[0], state)


@pytest.mark.parametrize("kind", ["f16d", "bf16d", "f16d-sr", "bf16d-sr", "mixed"])
@pytest.mark.parametrize("nx,ny", [(256, 40), (264, 33)])
def test_small_flow_batches_equal_solo_grids(lbm, kind, nx, ny):
    """Few grids whose strips of 240 columns are badly filled (one column beyond a strip
    of single steps too): the flow schedule steps them one step at a time."""
    def make(k):
        st = ("f32" if k % 2 else "f16d") if kind == "mixed" else kind
        g = lbm.Grid(nx, ny, 0.6 + 0.1 * k, 0.2, st.replace("-sr", ""))
        if st.endswith("-sr"):
            g.set_rounding("stochastic")
        g.init(*workloads.fourier_modes(nx, ny, amp=1e-2, seed=k))
        return g

    limits = [5, 12, 9]
    grids = [make(k) for k in range(3)]
    b = lbm.Batch(grids)
    b.set_schedule("flow")
    b.step(12, limits)
    b.step(3)
    assert b.sync() == 0
    got = [g.get_state()[0] for g in grids]
    b.close()
    for g in grids:
        g.close()
    for k, state in enumerate(got):
        with make(k) as h:
            for _ in range(limits[k] + 3):
                h.step(1)
            assert np.array_equal(h.get_state()[0], state)
