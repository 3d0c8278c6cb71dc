"""Which batches take passes of several steps (lbm_batch_get_pass), among them the ones
that the bitwise comparisons with single steps rely on; heights as built."""
import ctypes

import numpy as np
import pytest

import test_gpu_batch_pairs
from paper_0707_2437_gb300 import workloads

pytestmark = pytest.mark.gpu


def _batch(lbm, kind, lens):
    n = len(test_gpu_batch_pairs.SIZES)
    grids = [test_gpu_batch_pairs._grid(lbm, kind, lens, k) for k in range(n)]
    return grids, lbm.Batch(grids)


def _close(b, grids):
    b.close()
    for g in grids:
        g.close()


def test_bad_arguments(lbm):
    lib = lbm.load()
    n = ctypes.c_int()
    assert lib.lbm_batch_get_pass(None, 0, ctypes.byref(n)) == -1
    with lbm.Grid(16, 16, 0.8, 0.2) as g:
        b = lbm.Batch([g])
        assert lib.lbm_batch_get_pass(b.b, 0, None) == -1
        for k in (-1, 1):
            assert lib.lbm_batch_get_pass(b.b, k, ctypes.byref(n)) == -1
        b.close()


@pytest.mark.parametrize("kind,lens,steps", [("f32", False, 2), ("f32", True, 2),
                                             ("f16d", False, 1), ("bf16d", True, 1),
                                             ("f16d-sr", False, 1), ("mixed", False, 1)])
def test_passes_of_the_pair_tests(lbm, kind, lens, steps):
    """Those tests compare passes in FP32.  In 16 bits one of their widths is no multiple
    of eight: the batch is of two kinds and steps singly (passes: below)."""
    grids, b = _batch(lbm, kind, lens)
    assert {b.steps_per_pass(k) for k in range(len(grids))} == {steps}
    b.set_schedule("flow")
    assert {b.steps_per_pass(k) for k in range(len(grids))} == {steps}
    if steps == 2:
        b.set_config(1, 0)  # (heights of one row become four, the reach of a pass)
        assert b.get_config()["rows"] == 4
    _close(b, grids)


def _compare(lbm, make, sizes, limits, schedule, steps, looked_at):
    grids = [make(k) for k in range(len(sizes))]
    b = lbm.Batch(grids)
    b.set_schedule(schedule)
    assert {b.steps_per_pass(k) for k in range(len(grids))} == {steps}
    b.step(12, limits)
    b.step(3)
    assert b.sync() == 0
    got = {k: grids[k].get_state()[0] for k in looked_at}
    _close(b, grids)
    for k, state in got.items():
        with make(k) as h:
            for _ in range(min(12, limits[k]) + 3):
                h.step(1)
            assert np.array_equal(h.get_state()[0], state), sizes[k]


def _maker(lbm, sizes, kinds, lens=False):
    def make(k):
        nx, ny = sizes[k]
        kind = kinds[k % len(kinds)]
        g = lbm.Grid(nx, ny, 0.6 + 0.02 * k, 0.1 + 0.01 * k, kind.replace("-sr", ""))
        if kind.endswith("-sr"):
            g.set_rounding("stochastic")
        if lens:
            g.set_c2_field(workloads.c2_lens(nx, ny, 0.2))
        g.init(*workloads.fourier_modes(nx, ny, amp=1e-2, seed=k))
        return g
    return make


@pytest.mark.parametrize("kind,lens", [("f16d", False), ("bf16d", False), ("f16d-sr", False),
                                       ("bf16d-sr", False), ("f16d", True), ("bf16d", True)])
def test_16_bit_passes_in_lockstep_equal_single_steps(lbm, kind, lens):
    """Grids wide enough not to share warps: one lane and a part of a strip beyond 240
    columns, whole strips, packed last strips; limits that leave one step and that end
    early."""
    sizes = [(136, 9), (240, 33), (248, 5), (256, 100), (488, 20), (1208, 41)]
    _compare(lbm, _maker(lbm, sizes, [kind], lens), sizes, [1, 2, 9, 12, 5, 12], "lockstep", 2,
             range(len(sizes)))


@pytest.mark.parametrize("kind", ["f16d", "bf16d", "f16d-sr", "bf16d-sr"])
def test_16_bit_passes_in_flow_equal_single_steps(lbm, kind):
    """Enough work for passes to be the faster: strips of a part of 240 columns."""
    sizes = [(200, 300 + k) for k in range(32)]
    limits = [1 + (5 * k) % 13 for k in range(32)]
    _compare(lbm, _maker(lbm, sizes, [kind]), sizes, limits, "flow", 2, (0, 1, 2, 5, 12, 31))


@pytest.mark.parametrize("kind", ["f16d", "bf16d", "f16d-sr", "bf16d-sr"])
def test_mixed_passes_in_flow_equal_single_steps(lbm, kind):
    """FP32 and one 16-bit kind, strips filled whole, two of them, and by one lane."""
    sizes = [(120, 4), (240, 33), (240, 7), (480, 20), (120, 100), (248, 50)]
    _compare(lbm, _maker(lbm, sizes, ["f32", kind]), sizes, [1, 2, 9, 12, 5, 13], "flow", 2,
             range(len(sizes)))


@pytest.mark.parametrize("schedule", ["lockstep", "flow"])
@pytest.mark.parametrize("kind", ["f32", "f16d", "bf16d-sr", "mixed"])
def test_calls_of_one_step_between_others(lbm, schedule, kind):
    """Calls of one step run on a list of single-step walks: mixed with longer calls, and
    with a grid's rounding or field changed in between (both lists are built again)."""
    sizes = [(120, 64), (240, 300), (240, 96), (480, 200)]
    make = _maker(lbm, sizes, ["f32", "f16d"] if kind == "mixed" else [kind])
    grids = [make(k) for k in range(len(sizes))]
    b = lbm.Batch(grids)
    b.set_schedule(schedule)
    b.step(5)
    for n in (1, 1, 4, 1):
        b.step(n)
    lens = workloads.c2_lens(*sizes[0], 0.2)
    if not kind.endswith("-sr"):
        grids[0].set_c2_field(lens)
    b.step(1)
    b.step(3, [1, 0, 3, 2])
    b.step(1, [0, 1, 1, 0])
    assert b.sync() == 0
    got = [(g.t, g.get_state()[0]) for g in grids]
    _close(b, grids)
    for k, (t, state) in enumerate(got):
        assert t == 13 + [1, 1, 4, 2][k]
        with make(k) as h:
            for n in range(t):
                if n == 12 and k == 0 and not kind.endswith("-sr"):
                    h.set_c2_field(lens)
                h.step(1)
            assert np.array_equal(h.get_state()[0], state), sizes[k]


def test_tall_batch_takes_three_steps(lbm):
    """The grids of the test of tall tiles in a batch."""
    grids = [lbm.Grid(nx, ny, 0.7, 0.2) for nx, ny in [(64, 100003), (124, 20001)]]
    b = lbm.Batch(grids)
    assert [b.steps_per_pass(k) for k in range(2)] == [3, 3]
    _close(b, grids)
