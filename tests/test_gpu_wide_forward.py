"""The hour-angle form's wide forward (passes of 128 LSTs) and its two-sky pass (Hessian-vector
products) against the FP64 sums, over LST steps, cells of 1 / q pixel and LST counts at the edges of a
16-column group, of a pass and of the two forms.

Bounds: those of the hour-angle form on the 7-antenna hexagon, its least accurate array (V 1e-5 after
refinement); the data know nothing of the sky, so gradients and products carry the error of V once."""
import numpy as np
import pytest

from paper_2504_07090_gb300 import synth

pytestmark = pytest.mark.gpu

# hex side, LSTs, RA cells (LST step 5 RA / (16 LSTs) pixels: 1, 2, 5/2, 3/4, 1/2), Dec cells
GEOMETRIES = [(2, 5, 16, 9), (2, 5, 32, 9), (2, 5, 40, 7), (2, 20, 48, 6), (3, 10, 32, 7), (2, 60, 96, 3), (2, 64, 0, 3),
              (2, 65, 104, 3), (2, 70, 112, 4), (3, 80, 256, 2), (2, 120, 192, 3), (2, 125, 200, 2), (2, 130, 208, 2),
              (2, 200, 320, 2), (6, 70, 112, 4)]


def _problem(side, nt, nr, nd):
    if nr:
        return synth.drift_scan_problem("wide", side, 2, 150e6, 153e6, nt, nd, nr, 16, 4, 20, 41)
    p = synth.drift_scan_problem("wide", side, 2, 150e6, 153e6, nt, nd, 96, 16, 4, 20, 41)
    p.lst_rad = p.lst_rad[0] + np.arange(nt) * (p.ra_max - p.ra_min) / 96 * 3     # a step of three pixels
    return p


def _outputs(p, prec):
    import torch
    from paper_2504_07090_gb300 import fm
    h = fm.ForwardModel(p, prec, sigma=1.0)
    if prec not in ("fp64", "fp32"):
        assert h.contraction_info()["form"] == "hour_angle"
    tr = synth.draw_truth(p)
    th = torch.tensor(tr.theta.astype(np.float32), device="cuda").to(h.dtype)
    h.set_data(torch.tensor(synth.random_data(p, 1e4, 3).astype(np.float32), device="cuda").to(h.dtype))
    v = torch.tensor((tr.theta * np.random.default_rng(4).standard_normal(h.n_params)).astype(np.float32), device="cuda")
    out = {"V": h.forward(th), "grad": h.chi2_grad(th)[1]}
    if p.n_ant < 64:
        out |= {"hvp": h.hvp(th, v.to(h.dtype), full=True), "gn": h.hvp(th, v.to(h.dtype), full=False)}
    out = {k: t.cpu().double() for k, t in out.items()}
    h.sync_status()
    h.close()
    return out


@pytest.mark.parametrize("geo", GEOMETRIES)
@pytest.mark.parametrize("prec", ["fp16x3", "bf16x3", "fp16x1"])
def test_wide_and_two_sky_passes_match_fp64(geo, prec):
    p = _problem(*geo)
    a, b = _outputs(p, prec), _outputs(p, "fp64" if p.n_ant < 64 else "fp32")
    bound = {"fp16x3": 1e-5, "bf16x3": 1e-5, "fp16x1": 1e-3}[prec]
    for k in a:
        err = float((a[k] - b[k]).norm() / b[k].norm())
        assert err < (bound if k == "V" else 10 * bound), (k, err)
