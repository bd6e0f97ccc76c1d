"""Handles of large arrays with little redundancy are made without comparing every baseline with every other: 256
antennas (32,640 baselines, one vector twice or none) within a second, where it took up to 2.5."""
import time

import numpy as np
import pytest

from paper_2504_07090_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("redundant", [0, 1])
def test_large_arrays_are_set_up_quickly(redundant):
    import torch
    from paper_2504_07090_gb300 import fm
    ant = 60.0 * np.random.default_rng(3).standard_normal((256, 3))
    if redundant:                                        # one vector twice
        ant[3] = ant[2] + ant[1] - ant[0]
    p = synth.drift_scan_problem("large", 7, 1, 150e6, 150e6, 2, 3, 29, 8, 4, 20, 41, ant_enu=ant)
    torch.zeros(1, device="cuda")
    fm.ForwardModel(synth.config("tiny"), "fp64").close()
    t0 = time.perf_counter()
    h = fm.ForwardModel(p, "fp64", sigma=1.0)
    took = time.perf_counter() - t0
    h.close()
    assert took < 1.0
