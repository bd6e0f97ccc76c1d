"""FP64 and FP32 contractions per distinct fringe against the per-baseline sum (FM_HA=0,
FM_HA_GROUPS=0), over the geometries that take another tile, LST class or group count.

Bounds: FP64 differs by the rounding of the phases (1e3 rad at 1e-16) and of sums of at most
2e4 terms: 1e-11.  FP32 V and gradients of either form are within 3e-6 / 5e-5 of the FP64 oracle
(the bounds of the direct form), so two of them are within twice that of each other."""
import numpy as np
import pytest

from paper_2504_07090_gb300 import synth

pytestmark = pytest.mark.gpu

# hex side, channels, LSTs, Dec and RA cells: LST step of 1, 2, 1/2, 3/2 and 3/4 pixel, one LST, more
# than 64 LSTs (several LST tiles and adjoint blocks), more than 256 cells, off the grid
GEOMETRIES = {
    "step1": (3, 3, 10, 7, 32), "step2": (2, 2, 5, 9, 32), "half": (2, 2, 30, 5, 48), "step3_2": (4, 2, 20, 5, 96),
    "step3_4": (3, 2, 20, 6, 48), "one": (2, 2, 1, 5, 33), "lst70": (2, 1, 70, 3, 224), "cells300": (2, 1, 5, 3, 304),
    "hex61": (5, 1, 5, 3, 32), "offgrid": (3, 6, 3, 7, 41), "offgrid_odd": (4, 5, 2, 5, 29),
}


def _problem(name):
    if name == "random":          # 9 antennas, no two baselines alike
        rng = np.random.default_rng(5)
        ant = np.column_stack([rng.uniform(-40, 40, 9), rng.uniform(-40, 40, 9), rng.uniform(-0.5, 0.5, 9)])
        return synth.drift_scan_problem(name, 2, 3, 150e6, 155e6, 5, 6, 16, 8, 4, 20, 29, ant_enu=ant)
    if name == "hex91":           # 91 antennas: 135 groups, several group tiles
        return synth.drift_scan_problem(name, 6, 1, 150e6, 150e6, 10, 3, 32, 8, 4, 20, 3)
    side, nf, nt, nd, nr = GEOMETRIES[name]
    return synth.drift_scan_problem(name, side, nf, 146e6, 155e6, nt, nd, nr, 8, 4, 20, 19)


def _outputs(p, prec, airy, monkeypatch, general):
    import torch
    from paper_2504_07090_gb300 import fm
    for k in ("FM_HA", "FM_HA_GROUPS"):
        monkeypatch.setenv(k, "0" if general else "1")
    h = fm.ForwardModel(synth.with_airy_beam(p) if airy else p, prec, sigma=1.0)
    tr = synth.draw_truth(p)
    th = torch.tensor(tr.theta, dtype=h.dtype, device="cuda")
    data = torch.tensor(synth.random_data(p, 1e4, 3), dtype=h.dtype, device="cuda")
    x = torch.tensor(np.random.default_rng(2).standard_normal(h.n_pix_total), dtype=h.dtype, device="cuda")
    h.set_data(data)
    v = torch.tensor(synth.random_vectors(h.n_params, 1, 4)[0], dtype=h.dtype, device="cuda")
    out = {"V": h.forward(th), "Vx": h.forward_pixels(x)}
    if p.n_ant < 64:              # the FP64 epilogues hold n_bl complex in shared memory several times over
        out |= {"grad": h.chi2_grad(th)[1], "hvp": h.hvp(th, v, full=True)}
    out = {k: t.cpu().double() for k, t in out.items()}
    h.sync_status()
    h.close()
    return out


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("name", [*GEOMETRIES, "random", "hex91", "step1-airy", "offgrid-airy"])
def test_distinct_fringes_match_per_baseline_sum(name, prec, monkeypatch):
    p, airy = _problem(name.split("-")[0]), name.endswith("-airy")
    a = _outputs(p, prec, airy, monkeypatch, False)
    b = _outputs(p, prec, airy, monkeypatch, True)
    bound = {"fp64": dict(V=1e-11, Vx=1e-11, grad=1e-11, hvp=1e-11),
             "fp32": dict(V=6e-6, Vx=6e-6, grad=1e-4, hvp=1e-4)}[prec]
    for k in a:
        err = float((a[k] - b[k]).norm() / b[k].norm())
        assert err < bound[k], (k, err)
