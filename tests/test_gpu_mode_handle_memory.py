"""FP32 handles in hour-angle modes hold no buffers of the distinct-fringe sums: with nothing redundant a handle takes the
same memory whether baselines are grouped (which admits those sums) or not, to a few allocation granules of 2 MB.
The sums' buffers would be 16.6 MB."""
import numpy as np
import pytest

from paper_2504_07090_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_ra", [32, 29])           # the LST step a number of pixels and not
def test_mode_handles_hold_no_other_forms_buffers(n_ra, monkeypatch):
    import torch
    from paper_2504_07090_gb300 import fm
    ant = synth.hex_array(4)[:23] + 0.5 * np.random.default_rng(7).standard_normal((23, 3)) * [1.0, 1.0, 0.1]
    p = synth.drift_scan_problem("memory", 4, 64, 150e6, 153e6, 64, 3, n_ra, 8, 4, 20, 41, ant_enu=ant)
    p.lst_rad = p.lst_rad[0] + np.arange(64) * (np.deg2rad(48.0) / 32 / 4 if n_ra == 32 else 4.1e-3)

    def taken():
        free = torch.cuda.mem_get_info()[0]
        h = fm.ForwardModel(p, "fp32", sigma=1.0)
        n = free - torch.cuda.mem_get_info()[0]
        assert h.mode_table_bytes() > 0
        h.close()
        return n

    taken()
    got = []
    for groups in ("1", "0"):
        monkeypatch.setenv("FM_HA_GROUPS", groups)
        got.append(taken())
    assert abs(got[0] - got[1]) <= 3 << 21, got
