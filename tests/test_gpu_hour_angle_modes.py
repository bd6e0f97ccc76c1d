"""The contraction in hour-angle modes (split precisions, Gaussian beam) against the FP64 per-baseline sum, over
LSTs on and off the pixel grid, in and out of order, and sizes at the edges of its tiles: 1 and odd numbers of
declinations and more than 64 of them, LST counts around 16 and 64, groups past 64 and modes past 128.

Bounds: those of the split forms on the 7-antenna hexagon (V 1e-5); the data know nothing of the sky, so
gradients and products carry the error of V once."""
import numpy as np
import pytest

from paper_2504_07090_gb300 import synth

pytestmark = pytest.mark.gpu

# hex side, channels, LSTs, Dec and RA cells, LST pattern
GEOMETRIES = {
    "step1": (3, 3, 10, 7, 32, None), "half": (2, 2, 30, 5, 48, None), "one_lst": (2, 2, 1, 5, 33, None),
    "one_dec": (2, 2, 17, 1, 40, None), "lst70": (2, 1, 70, 3, 224, None), "dec130": (2, 1, 5, 130, 32, None),
    "hex61": (5, 1, 5, 3, 32, None), "offgrid": (3, 6, 3, 7, 41, None), "offgrid16": (4, 3, 16, 6, 70, None),
    "uneven": (4, 2, 9, 5, 64, "uneven"), "backwards": (3, 2, 6, 5, 64, "backwards"), "wide_lst": (2, 2, 65, 4, 100, "uneven"),
    "hex127": (7, 1, 120, 3, 384, None), "turn": (3, 2, 6, 5, 64, "turn"),
}


def _problem(name):
    side, nf, nt, nd, nr, lst = GEOMETRIES[name]
    p = synth.drift_scan_problem(name, side, nf, 146e6, 155e6, nt, nd, nr, 16, 4, 20, 19)
    if lst == "uneven":
        p.lst_rad = p.lst_rad + 1e-3 * np.random.default_rng(8).standard_normal(nt)
    if lst == "backwards":
        p.lst_rad = np.ascontiguousarray(p.lst_rad[::-1])
    if lst == "turn":             # hour angles around -2 pi: right ascensions a turn ahead of the LSTs
        p.ra_min, p.ra_max = p.ra_min + 2 * np.pi, p.ra_max + 2 * np.pi
    return p


def _outputs(p, prec):
    import torch
    from paper_2504_07090_gb300 import fm
    h = fm.ForwardModel(p, prec, sigma=1.0)
    assert (h.mode_table_bytes() > 0) == (prec != "fp64")
    th = torch.tensor(synth.draw_truth(p).theta.astype(np.float32), device="cuda").to(h.dtype)
    h.set_data(torch.tensor(synth.random_data(p, 1e4, 3).astype(np.float32), device="cuda").to(h.dtype))
    x = np.random.default_rng(2).standard_normal(h.n_pix_total).astype(np.float32)
    v = synth.random_vectors(h.n_params, 1, 4)[0].astype(np.float32)
    out = {"V": h.forward(th), "Vx": h.forward_pixels(torch.tensor(x, device="cuda").to(h.dtype))}
    if p.n_ant < 64:              # the FP64 epilogues hold n_bl complex in shared memory several times over
        v = torch.tensor(v, device="cuda").to(h.dtype)
        out |= {"grad": h.chi2_grad(th)[1], "hvp": h.hvp(th, v, full=True), "gn": h.hvp(th, v, full=False)}
    out = {k: t.cpu().double() for k, t in out.items()}
    h.sync_status()
    h.close()
    return out


@pytest.mark.parametrize("prec", ["fp16x3", "bf16x3", "fp32"])
@pytest.mark.parametrize("name", list(GEOMETRIES))
def test_hour_angle_modes_match_fp64(name, prec, monkeypatch):
    p = _problem(name)
    a = _outputs(p, prec)
    for k in ("FM_HA", "FM_HA_GROUPS"):
        monkeypatch.setenv(k, "0")
    b = _outputs(p, "fp64")
    for k in a:
        err = float((a[k] - b[k]).norm() / b[k].norm())
        assert err < (1e-5 if k in ("V", "Vx") else 1e-4), (k, err)


# The mass matrix from fewer maps than LSTs against the responses of every LST: both form FP32 responses from FP16
# split transforms and agree to 2e-6 (the bound of the drift-scan cell image's test).
@pytest.mark.parametrize("name", ["half", "one_dec", "lst70", "offgrid16", "uneven", "wide_lst"])
@pytest.mark.parametrize("block", [64, 1])
def test_mass_matrix_from_hour_angle_maps(name, block, monkeypatch):
    import torch
    from paper_2504_07090_gb300 import fm
    p = _problem(name)
    tr = synth.draw_truth(p)
    mu, lam = (torch.tensor(a.astype(np.float32), device="cuda") for a in synth.prior_for(p, tr.theta))
    got = []
    for ha in ("1", "0"):
        monkeypatch.setenv("FM_HA", ha)
        h = fm.ForwardModel(p, "fp16x3", sigma=50.0)
        th = torch.tensor(tr.theta.astype(np.float32), device="cuda")
        h.set_data(torch.tensor(synth.random_data(p, 1e3, 7).astype(np.float32), device="cuda"))
        h.set_prior(mu, lam)
        h.build_precond(th, block)
        got.append(h.precond_blocks().cpu().numpy()[: p.n_sky_params * block])
        h.close()
    assert np.linalg.norm(got[0] - got[1]) < 2e-6 * np.linalg.norm(got[1])
