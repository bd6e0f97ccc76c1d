"""Grids whose hour angles stay off the meridian, where the beam's maximum lies in the cells around the grid: visibilities
and sky gradients of every channel against the FP64 per-baseline sum.

Bounds per channel: FP32 V 3e-6 and gradient 5e-5, FP16 split 1e-5 and 1e-4, BF16 split 2e-5 and 2e-4 (the forms'
own); the data know nothing of the sky, so the gradient carries the error of the responses once.  The FP16 split has
a fixed scale, 2^-38 of a response at the beam's maximum (6e-8 / 2^14): it is asked only where the nearest cell keeps
1e-4 of the beam."""
import numpy as np
import pytest

from paper_2504_07090_gb300 import synth

pytestmark = pytest.mark.gpu

BOUND = {"fp32": (3e-6, 5e-5), "fp16x3": (1e-5, 1e-4), "bf16x3": (2e-5, 2e-4)}


# RA cells, degrees a cell, LSTs, FWHM at 150 MHz (degrees); degrees off the meridian; where the FP16 split ends
GRIDS = [((13, 1.9, 4, 5.0), (0, 14, -16, 18, 20, 22, 25, -27), 23), ((12, 3.0, 4, 8.0), (0, 28, 31, 34, 38), 35),
         ((16, 1.0, 4, 3.0), (0, 11, 12.5, -14, 15.5), 14.5), ((16, 1.1, 4, 10.0), (0, 25, 35), 30)]


def _problem(grid, off_deg):
    n_ra, cell_deg, n_lst, fwhm = grid
    p = synth.drift_scan_problem("off", 2, 2, 120e6, 180e6, n_lst, 12, n_ra, 8, 4, 20, 19)
    cell = np.deg2rad(cell_deg)
    p.ra_min, p.ra_max = 0.3, 0.3 + n_ra * cell
    p.lst_rad = 0.3 + 0.5 * n_ra * cell + np.deg2rad(off_deg) + (np.arange(n_lst) - 0.5 * (n_lst - 1)) * cell
    p.beam_fwhm_ref_rad = np.deg2rad(fwhm)
    return p


def _outputs(p, prec):
    import torch
    from paper_2504_07090_gb300 import fm
    h = fm.ForwardModel(p, prec, sigma=1.0)
    th = torch.tensor(synth.draw_truth(p).theta.astype(np.float32), device="cuda").to(h.dtype)
    h.set_data(torch.tensor(synth.random_data(p, 1e4, 3).astype(np.float32), device="cuda").to(h.dtype))
    table = h.mode_table_bytes()
    V, g = h.forward(th), h.chi2_grad(th)[1][: p.n_sky_params]
    out = [t.cpu().double().reshape(p.n_freq, -1) for t in (V, g)]
    h.sync_status()
    h.close()
    return out, table


@pytest.mark.parametrize("grid,off,prec", [(g, o, q) for g, offs, last in GRIDS for o in offs for q in BOUND
                                           if q != "fp16x3" or abs(o) < last])
def test_off_meridian_grids_match_fp64(grid, off, prec, monkeypatch):
    p = _problem(grid, off)
    a, table = _outputs(p, prec)
    assert off or table > 0
    for k in ("FM_HA", "FM_HA_GROUPS"):
        monkeypatch.setenv(k, "0")
    b, _ = _outputs(p, "fp64")
    for x, y, bound in zip(a, b, BOUND[prec]):
        err = (x - y).norm(dim=1) / y.norm(dim=1)
        assert float(err.max()) < bound, err
