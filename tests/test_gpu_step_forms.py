"""Which form step calls take (lbm_get_step_form).  The tests that compare passes of
several steps and resident launches with single steps, bit for bit, say something only
where those forms run, so their sizes are looked at here."""
import ctypes

import numpy as np
import pytest

import test_gpu_resident
import test_gpu_step_pairs
from paper_0707_2437_gb300 import workloads

pytestmark = pytest.mark.gpu


def _grid(lbm, nx, ny, kind, option=""):
    g = lbm.Grid(nx, ny, 0.7, 0.2, kind.replace("-sr", ""))
    if kind.endswith("-sr"):
        g.set_rounding("stochastic")
    if option == "field":
        g.set_c2_field(workloads.c2_lens(nx, ny, 0.2))
    if option == "drive":
        g.set_drive(1e-3, 40.0)
    return g


def test_bad_arguments(lbm):
    lib = lbm.load()
    assert lib.lbm_get_step_form(None, 1, None, None) == -1
    with lbm.Grid(16, 16, 0.8, 0.2) as g:
        assert lib.lbm_get_step_form(g.h, 0, None, None) == -1
        assert lib.lbm_get_step_form(g.h, 5, None, None) == 0
        steps = ctypes.c_int()
        assert lib.lbm_get_step_form(g.h, 1 << 40, None, ctypes.byref(steps)) == 0
        assert steps.value == 0x7fffffff


@pytest.mark.parametrize("kind,lens", [("f32", False), ("f32", True), ("f16d", False),
                                       ("bf16d", True), ("f16d-sr", False), ("bf16d-sr", False)])
@pytest.mark.parametrize("shape", range(4))
def test_shapes_of_the_pair_tests_take_passes(lbm, kind, lens, shape):
    """All but one: FP32 with a c2 field is faster in single steps at a width of four.
    One is small enough for its long calls to run resident; short ones take passes."""
    nx, ny = test_gpu_step_pairs.SHAPES["f32" if kind == "f32" else "16"][shape]
    with _grid(lbm, nx, ny, kind, "field" if lens else "") as g:
        form, steps = g.step_form(3)
        assert form == "launches"
        assert (steps > 1) == (not (kind == "f32" and lens and nx == 4)), steps
        assert (g.step_form(100)[0] == "resident") == (nx * ny < 300000)
        assert g.step_form(1) == ("launches", 1)
        g.set_config(1, 8, 4)
        assert g.step_form(100) == ("launches", 1)


@pytest.mark.parametrize("kind,nx,ny", [
    ("f32", 119, 12001), ("f32", 239, 9001), ("f32", 601, 4001), ("f32", 1001, 1601),
    ("f16d", 238, 9001), ("f16d", 1202, 3001), ("bf16d", 478, 9001),
    ("bf16d-sr", 238, 15001), ("f16d-sr", 1202, 5001)])
def test_ragged_widths_of_the_pair_tests_take_passes(lbm, kind, nx, ny):
    with _grid(lbm, nx, ny, kind) as g:
        assert g.step_form(35) == ("launches", 2)


@pytest.mark.parametrize("nx,ny,steps", [(60, 50021, 3), (1012, 4003, 2), (1012, 12001, 3)])
def test_steps_of_a_pass_with_a_c2_field(lbm, nx, ny, steps):
    """Part of a strip; nine whole strips and a narrow one, in passes of two steps and,
    on the taller grid (nine strips of 112 columns and one of four), of three: those
    states are compared here."""
    with _grid(lbm, nx, ny, "f32", "field") as g:
        assert g.step_form(14) == ("launches", steps)
        if (nx, ny) != (1012, 12001):
            return
        fields = workloads.fourier_modes(nx, ny, amp=1e-2, seed=nx + ny)
        g.init(*fields)
        for n in (3, 8, 1, 2):
            g.step(n)
        state = g.get_state()[0]
        g.init(*fields)
        for _ in range(14):
            g.step(1)
        assert np.array_equal(g.get_state()[0], state)


@pytest.mark.parametrize("nx,ny", test_gpu_resident.SIZES)
@pytest.mark.parametrize("kind,option", [("f32", ""), ("f32", "field"), ("f32", "drive"),
                                         ("f16d", ""), ("bf16d", "field"), ("f16d-sr", ""),
                                         ("bf16d-sr", "drive")])
def test_sizes_of_the_resident_tests_run_resident(lbm, nx, ny, kind, option):
    """Their long calls do, but for the largest grid with stochastic rounding (every
    site is hashed there, every pair of sites in the step kernel)."""
    if option == "drive" and nx < 4:
        pytest.skip("a driven channel needs nx >= 4")
    with _grid(lbm, nx, ny, kind, option) as g:
        if (nx, ny) == (600, 590) and kind.endswith("-sr"):
            return
        assert g.step_form(150) == ("resident", 150)
        assert g.step_form(1) == ("launches", 1)
        g.set_persistent(False)
        assert g.step_form(150)[0] == "launches"


@pytest.mark.parametrize("kind,option,nx,ny,n,resident", [
    ("f32", "", 64, 64, 4, True), ("f32", "", 509, 381, 4, True), ("f32", "", 640, 640, 4, False),
    ("f32", "", 640, 640, 64, True), ("f32", "field", 512, 512, 4, False),
    ("f32", "field", 512, 512, 64, True), ("f32", "field", 640, 640, 512, False),
    ("f16d", "", 256, 256, 4, True), ("f16d", "", 512, 512, 4, False),
    ("f16d", "", 512, 512, 16, True), ("bf16d", "", 640, 640, 512, False),
    ("f16d", "drive", 640, 640, 64, True), ("bf16d", "field", 600, 600, 6, False),
    ("f16d-sr", "", 256, 256, 8, True), ("f16d-sr", "", 512, 512, 4, False),
    ("bf16d-sr", "", 600, 600, 512, False)])
def test_resident_where_it_is_the_faster(lbm, kind, option, nx, ny, n, resident):
    """Both sides of the line, at sizes where the two forms differ by a tenth or more."""
    with _grid(lbm, nx, ny, kind, option) as g:
        assert (g.step_form(n)[0] == "resident") == resident


def test_small_grids_on_several_streams(lbm):
    """Grids of 256^2 take turns on the SMs when they run resident: on eight streams
    their step launches overlap instead.  Grids of one tile have an SM each, and a large
    grid's stream does not count."""
    streams = [lbm.new_stream() for _ in range(8)]
    big = lbm.Grid(2048, 2048, 0.8, 0.2, stream=lbm.new_stream())
    grids = [lbm.Grid(256, 256, 0.8, 0.2, stream=s) for s in streams]
    tiny = lbm.Grid(16, 16, 0.8, 0.2, stream=streams[0])
    fields = workloads.fourier_modes(256, 256, amp=1e-2, seed=1)
    for g in grids:
        g.init(*fields)
        assert g.step_form(100)[0] == "launches"
        g.step(100)
    assert tiny.step_form(100)[0] == "resident"
    for g in grids[1:4]:
        g.close()
    for g in grids[4:]:
        g.set_stream(streams[0])
    rest = [grids[0]] + grids[4:]
    for g in rest:
        assert g.step_form(100)[0] == "resident"
        g.step(20)
    states = [g.get_state()[0] for g in rest]
    for g in rest + [tiny, big]:
        g.close()
    with lbm.Grid(256, 256, 0.8, 0.2) as h:
        h.set_persistent(False)
        h.init(*fields)
        h.step(120)
        assert all(np.array_equal(h.get_state()[0], s) for s in states)


def test_forms_under_settings(lbm):
    with lbm.Grid(256, 256, 0.8, 0.2) as g:
        g.set_persistent(True)
        assert g.step_form(64) == ("persistent", 64)
        assert g.step_form(63)[0] == "launches"
        g.set_persistent("auto")
        g.set_timing(True)
        assert g.step_form(64) == ("launches", 1)
        g.set_timing(False)
        g.set_gradient("forward")
        assert g.step_form(64) == ("launches", 1)
    with lbm.Slab(256, 64, 0.8, 0.2) as s:
        assert s.step_form(1) == ("persistent", 1)


@pytest.mark.parametrize("nx,ny", [(64, 64), (2048, 1025)])
def test_first_step_call_under_capture(lbm, nx, ny):
    """Plans are made by the first call that needs them, which may be one into a stream
    that is being captured: launches of the step kernel, single or passes, that a replay
    repeats."""
    import torch
    fields = workloads.fourier_modes(nx, ny, amp=1e-2, seed=nx)
    stream = torch.cuda.Stream()
    with lbm.Grid(nx, ny, 0.7, 0.2, stream=stream) as warm:  # (kernels are loaded)
        warm.init(*fields)
        warm.step(1)
        warm.step(7)
        warm.sync()
    with lbm.Grid(nx, ny, 0.7, 0.2, stream=stream) as g:
        g.init(*fields)
        g.sync()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            assert g.step_form(7)[0] == "launches"
            g.step(7)
        with torch.cuda.stream(stream):
            graph.replay()
        state = g.get_state()[0]
        g.set_persistent(False)
        g.init(*fields)
        for _ in range(7):
            g.step(1)
        assert np.array_equal(g.get_state()[0], state)
