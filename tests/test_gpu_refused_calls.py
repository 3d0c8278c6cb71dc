"""Calls of the CUDA runtime that fail leave the library usable: the failure is an error
of the call that met it or, where there is another way, no error at all.  The failures
are made on the host, by a library preloaded into a child process (fake_cuda.c) that
answers the call instead of the runtime; nothing invalid reaches the GPU.  States are
compared bit for bit with grids that met no failure."""
import os
import subprocess
import sys
import textwrap

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

HEAD = """
    import ctypes
    import numpy as np
    from paper_0707_2437_gb300 import lbm, workloads
    fake = ctypes.CDLL(None)
    malloc = ctypes.c_int.in_dll(fake, "fake_malloc")
    group = ctypes.c_int.in_dll(fake, "fake_group")

    def grid(nx, ny, storage="f32"):
        g = lbm.Grid(nx, ny, 0.7, 0.2, storage)
        g.init(*workloads.fourier_modes(nx, ny, amp=1e-2, seed=nx + ny))
        return g

    def alone(nx, ny, n, storage="f32"):
        with grid(nx, ny, storage) as g:
            g.set_persistent(False)
            g.step(n)
            return g.get_state()[0]
"""


@pytest.fixture(scope="module")
def fake_lib(lbm, tmp_path_factory):
    so = str(tmp_path_factory.mktemp("fake") / "fake_cuda.so")
    src = os.path.join(ROOT, "tests", "fake_cuda.c")
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    subprocess.run(["gcc", "-shared", "-fPIC", "-O1", "-I", os.path.join(cuda, "include"), src,
                    "-o", so, "-ldl"], check=True)
    return so


def _run(fake_lib, body):
    env = dict(os.environ, LD_PRELOAD=fake_lib, PYTHONPATH=ROOT)
    code = textwrap.dedent(HEAD) + textwrap.dedent(body)
    r = subprocess.run([sys.executable, "-c", code], env=env, cwd=ROOT, timeout=300,
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr


@pytest.mark.parametrize("change", ["set_schedule('flow')", "set_config(8, 0)",
                                    "set_walk16('v4')"])
def test_failed_work_list_is_built_again_by_the_next_step(fake_lib, change):
    """A change whose work-list cannot be allocated fails, a step call while that lasts
    fails too and steps nothing, and later ones run under the new setting."""
    _run(fake_lib, f"""
        sizes = [(64, 40, "f16d"), (120, 33, "f32")]
        grids = [grid(*s) for s in sizes]
        b = lbm.Batch(grids)
        b.step(3)
        malloc.value = 1
        for call in (lambda: b.{change}, lambda: b.step(3)):
            try:
                call()
            except lbm.LbmError as e:
                assert e.status == lbm.LBM_ENOMEM, e
            else:
                raise AssertionError("no error")
        assert [g.t for g in grids] == [3, 3]
        malloc.value = 0
        b.step(4)
        assert b.sync() == 0
        for g, (nx, ny, st) in zip(grids, sizes):
            assert g.t == 7
            assert np.array_equal(g.get_state()[0], alone(nx, ny, 7, st))
    """)


@pytest.mark.parametrize("schedule", ["lockstep", "flow"])
def test_failed_list_for_calls_of_one_step(fake_lib, schedule):
    """Calls of one step have a list of their own, made by the first of them; where it
    cannot be allocated that call fails, and others run."""
    _run(fake_lib, f"""
        sizes = [(120, 40), (116, 33), (240, 64)]
        grids = [grid(*s) for s in sizes]
        b = lbm.Batch(grids)
        b.set_schedule("{schedule}")
        assert b.steps_per_pass() == 2
        b.step(4)
        malloc.value = 1
        try:
            b.step(1)
        except lbm.LbmError as e:
            assert e.status == lbm.LBM_ENOMEM, e
        else:
            raise AssertionError("no error")
        b.step(4)
        malloc.value = 0
        b.step(1)
        b.step(4)
        b.step(1)
        assert b.sync() == 0
        for g, s in zip(grids, sizes):
            assert g.t == 14
            assert np.array_equal(g.get_state()[0], alone(*s, 14))
    """)


@pytest.mark.parametrize("nx,ny,tiles", [(400, 4, "one cluster"), (256, 256, "all SMs")])
def test_refused_resident_launch_steps_by_the_step_kernel(fake_lib, nx, ny, tiles):
    """A stream that owns too few SMs for a grid's tiles still steps it: the call whose
    launch is refused, the next one, and one after the grid has moved to a stream that
    takes such launches."""
    _run(fake_lib, f"""
        g = grid({nx}, {ny})
        g.step(10)
        group.value = 1
        g.step(11)
        g.step(12)
        g.sync()
        assert g.t == 33
        assert np.array_equal(g.get_state()[0], alone({nx}, {ny}, 33)), "{tiles}"
        group.value = 0
        g.set_stream(lbm.new_stream())
        g.step(13)
        assert np.array_equal(g.get_state()[0], alone({nx}, {ny}, 46))
    """)
