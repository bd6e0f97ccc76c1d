"""Mass-matrix build: the drift-scan cell image against the fringes of every LST, and the panel
Cholesky of the gain block against numpy, at sizes below, at and between the panel width.

Bounds: the two routes form the same FP32 responses up to the rounding of a cell's direction (6e-8 of
phases below 64 turns, 2e-5 at most at one pixel, averaged over the pixels): the blocks agree to 2e-6.
p = L z with an FP64 factor, stored as FP32: 1e-6."""
import numpy as np
import pytest

from paper_2504_07090_gb300 import synth

pytestmark = pytest.mark.gpu


def _handle(p, prec, seed=7):
    import torch
    from paper_2504_07090_gb300 import fm
    h = fm.ForwardModel(p, prec, sigma=50.0)
    tr = synth.draw_truth(p)
    th = torch.tensor(tr.theta, dtype=h.dtype, device="cuda")
    h.set_data(torch.tensor(synth.random_data(p, 1e3, seed), dtype=h.dtype, device="cuda"))
    mu, lam = synth.prior_for(p, tr.theta)
    h.set_prior(torch.tensor(mu, dtype=h.dtype, device="cuda"), torch.tensor(lam, dtype=h.dtype, device="cuda"))
    return h, th


# side, channels, LSTs, Dec and RA cells: steps of 1, 2, 4, 1/2, 3/2, 3/4 pixel, RA cells no multiple of 4, one LST
@pytest.mark.parametrize("geo", [(4, 2, 10, 7, 32), (2, 2, 5, 9, 32), (2, 2, 5, 9, 64), (2, 2, 30, 5, 48),
                                 (3, 2, 20, 5, 96), (2, 2, 20, 6, 48), (2, 1, 40, 5, 126), (2, 2, 1, 5, 32)])
@pytest.mark.parametrize("block", [64, 1])
@pytest.mark.parametrize("airy", [False, True])
def test_cell_image_matches_fringes_of_every_lst(geo, block, airy, monkeypatch):
    side, nf, nt, nd, nr = geo
    p = synth.drift_scan_problem("mass", side, nf, 148e6, 152e6, nt, nd, nr, 16, 8, 20, 3)
    p = synth.with_airy_beam(p) if airy else p
    got = []
    for ha in ("1", "0"):
        monkeypatch.setenv("FM_HA", ha)
        h, th = _handle(p, "fp16x3")
        h.build_precond(th, block)
        got.append(h.precond_blocks().cpu().numpy()[: p.n_sky_params * block])
        h.close()
    assert np.linalg.norm(got[0] - got[1]) < 2e-6 * np.linalg.norm(got[1])


@pytest.mark.parametrize("n_ant, n_gain", [(2, 1), (3, 4), (4, 4), (5, 4), (7, 4), (19, 4), (37, 4)])
@pytest.mark.parametrize("prec", ["fp16x3", "fp64"])
def test_gain_factor_matches_numpy(n_ant, n_gain, prec):
    import torch
    p = synth.drift_scan_problem("gain", 4, 4, 148e6, 152e6, 5, 5, 32, 16, 4, 20, 3, n_gain=n_gain)
    p.ant_enu = np.ascontiguousarray(p.ant_enu[:n_ant])
    h, th = _handle(p, prec)
    h.build_precond(th, 64)
    ng = 2 * n_ant * n_gain
    H = h.precond_blocks().cpu().numpy()[-ng * ng:].reshape(ng, ng)
    L = np.linalg.cholesky(H)
    z = np.random.default_rng(3).standard_normal(h.n_params)
    p0 = h.precond_apply(0, torch.tensor(z, dtype=h.dtype, device="cuda"))
    back = h.precond_apply(1, p0).cpu().double().numpy()
    zg = z[-ng:] if prec == "fp64" else z[-ng:].astype(np.float32).astype(float)
    want = L @ zg
    assert np.linalg.norm(p0.cpu().double().numpy()[-ng:] - want) < 1e-6 * np.linalg.norm(want)
    # L^-1 L z: the rounding of p times the factor's condition number
    assert np.linalg.norm(back[-ng:] - zg) < 1e-7 * np.linalg.cond(L) * np.linalg.norm(zg)
    h.close()
