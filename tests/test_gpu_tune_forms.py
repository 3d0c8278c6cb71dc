"""The tuner keeps the forms of step calls that are faster than single steps: a tuned
grid must not step more slowly than an untuned one, whatever the cache file held."""
import json

import numpy as np
import pytest

from paper_0707_2437_gb300 import workloads

pytestmark = pytest.mark.gpu


def _grid(lbm, nx, ny, storage="f32"):
    g = lbm.Grid(nx, ny, 0.7, 0.2, storage)
    g.init(*workloads.fourier_modes(nx, ny, amp=1e-2, seed=nx + ny))
    return g


@pytest.mark.parametrize("nx,ny,storage,form", [(400, 4, "f32", "resident"),
                                                (128, 96, "f16d", "resident"),
                                                (1536, 2048, "f32", "launches")])
def test_tuned_grid_keeps_the_faster_form(lbm, nx, ny, storage, form):
    with _grid(lbm, nx, ny, storage) as g, _grid(lbm, nx, ny, storage) as h:
        assert g.step_form(100)[0] == form
        g.step(5)
        state = g.get_state()[0]
        g.tune()
        assert np.array_equal(g.get_state()[0], state) and g.t == 5
        assert g.step_form(100)[0] == form
        if form == "launches":
            assert g.step_form(100)[1] > 1
        g.step(37)
        h.step(42)
        assert np.array_equal(g.get_state()[0], h.get_state()[0])


@pytest.mark.parametrize("numbers", [4, 5])
@pytest.mark.parametrize("nx,ny,form", [(400, 4, "resident"), (1536, 2048, "launches")])
def test_entry_without_the_forms(lbm, tmp_path, nx, ny, form, numbers):
    """Files of earlier versions hold a tile configuration and no word of the forms, or
    a fifth number that could be zero because nothing was timed: the configuration is
    taken, the forms are timed and the entry is completed."""
    cache = tmp_path / "tune.json"
    with _grid(lbm, nx, ny) as g:
        g.tune(str(cache))
    key, entry = next(iter(json.loads(cache.read_text()).items()))
    assert len(entry) == 6
    cache.write_text(json.dumps({key: [2, 8, 4, 0, 0][:numbers]}))
    with _grid(lbm, nx, ny) as g:
        assert g.tune(str(cache)) == (2, 8, 4, 0)
        got = g.step_form(100)
        assert got[0] == form and got[1] > 1
    assert json.loads(cache.read_text()) == {key: [2, 8, 4, 0] + entry[4:]}


def test_options_are_tuned_by_themselves(lbm, tmp_path):
    """A driven grid steps once a launch; that says nothing of a plain grid of its size.
    A grid with a c2 field does not meet the configuration of one without."""
    cache = str(tmp_path / "tune.json")
    nx, ny = 1536, 1024
    with _grid(lbm, nx, ny, "f16d") as g:
        g.set_drive(1e-3, 500.0)
        g.tune(cache)
        assert g.step_form(100) == ("launches", 1)
    with _grid(lbm, nx, ny, "f16d") as g, _grid(lbm, nx, ny, "f16d") as h:
        form = h.step_form(100)
        g.tune(cache)
        assert g.step_form(100) == form
    with _grid(lbm, nx, ny, "f16d") as g:
        g.set_c2_field(workloads.c2_lens(nx, ny, 0.2))
        g.tune(cache)
    assert len(json.load(open(cache))) == 3
