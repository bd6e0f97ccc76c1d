"""The launch-grid tuner beside handles that compute in hour-angle modes, whose kernels do not use the grids: their
timings are kept apart from those of the same sizes in hour-angle cells, and no grid is chosen for them."""
from types import SimpleNamespace

import pytest

pytest.importorskip("torch")
from paper_2504_07090_gb300 import autotune  # noqa: E402


class Model:
    def __init__(self, modes):
        self.prob = SimpleNamespace(n_ant=37, n_freq=16, n_dec=32, n_ra=64, n_lst=20)
        self.precision, self.modes, self.grids, self.set = "fp16x3", modes, (152, 152), []

    def contraction_info(self):
        return {"form": "hour_angle", "fringes": 63, "lst_step_cells": 1, "hour_angle_cells": 128}

    def mode_table_bytes(self):
        return 1000 if self.modes else 0

    def set_launch_grids(self, f, a):
        self.set.append(f)
        self.grids = (f or 152, a or 152)

    def launch_grids(self):
        return self.grids


@pytest.fixture
def timed(monkeypatch):
    seen = []

    def measure(model, theta, candidates, reps):
        seen.append(model)
        return {"8": 2.0, "152": 1.0} if not model.modes else {"8": 1.0, "152": 1.0}
    monkeypatch.setattr(autotune, "measure", measure)
    return seen


def test_timings_of_modes_and_cells_are_kept_apart(tmp_path, timed):
    path = str(tmp_path / "grids.json")
    modes, cells = Model(True), Model(False)
    assert autotune.shape_key(modes) != autotune.shape_key(cells)
    autotune.shape_times([modes], [None], path)
    tables, n = autotune.shape_times([cells, modes], [None, None], path)
    assert n == 1 and timed == [modes, cells] and tables[0] == {"8": 2.0, "152": 1.0}


def test_a_batch_in_modes_is_stepped_once(tmp_path, timed):
    models, steps = [Model(True), Model(True)], []
    rep = autotune.tune_batch(models, [None, None], lambda: steps.append(1) or 5.0, cache_path=str(tmp_path / "g.json"))
    assert len(steps) == 1 and rep["slack"] == "default" and rep["ms_per_step"] == {"default": 5.0}
    assert all(m.grids == (152, 152) for m in models)


def test_only_models_that_use_grids_are_given_them(tmp_path, timed):
    modes, cells = Model(True), Model(False)
    ms = iter([5.0, 4.0, 3.0, 6.0])
    rep = autotune.tune_batch([modes, cells], [None, None], lambda: next(ms), slacks=(1.0, 2.0, 3.0),
                              cache_path=str(tmp_path / "g.json"))
    assert rep["slack"] == 2.0 and cells.grids == (8, 8) and modes.grids == (152, 152)
