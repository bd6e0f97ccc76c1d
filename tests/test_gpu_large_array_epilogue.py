"""The chi^2 epilogue of large arrays (residuals of a CTA only) against the FP32 per-baseline form, around the size
where it takes over (70 antennas) and at 127, on its fused route, after the finished forward and with the delay
filter.  Bounds: those of the split forms (chi^2 2e-5, gradient 1e-4), the data knowing nothing of the sky."""
import numpy as np
import pytest

from paper_2504_07090_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_ant", [69, 70, 127])
@pytest.mark.parametrize("route", ["fused", "finished", "filter"])
def test_large_array_epilogue_matches_per_baseline_form(n_ant, route, monkeypatch):
    import torch
    from paper_2504_07090_gb300 import fm
    p = synth.drift_scan_problem("large", 7, 3, 150e6, 153e6, 5, 3, 32, 16, 4, 20, 41, ant_enu=synth.hex_array(7)[:n_ant])
    th = synth.draw_truth(p).theta.astype(np.float32)
    d = synth.random_data(p, 1e4, 3).astype(np.float32)
    if route == "finished":
        monkeypatch.setenv("FM_HA_FUSED_CHI2", "0")
    out = []
    for prec, ha in (("fp16x3", "1"), ("fp32", "0")):
        monkeypatch.setenv("FM_HA", ha)
        h = fm.ForwardModel(p, prec, sigma=1.0)
        h.set_data(torch.tensor(d, device="cuda"))
        if route == "filter":
            h.set_delay_filter(250e-9, 1e-8)
        scal, grad = h.chi2_grad(torch.tensor(th, device="cuda"))
        out.append((float(scal[0]), grad.cpu().double()))
        h.sync_status()
        h.close()
    (ca, ga), (cb, gb) = out
    assert abs(ca - cb) < 2e-5 * cb
    n = p.n_sky_params if route == "filter" else None      # the filter removes what the gains' gradient contracts with
    assert float((ga[:n] - gb[:n]).norm() / gb[:n].norm()) < 1e-4
