"""The delay filter's matrix products at channel counts around its blocks of four and eight and its eight
warps of eight channels, against the oracle, with data that know nothing of the sky (so that what passes
the filter is of the data's size).  Bounds: those of the filter's FP64 / FP32 cases.  The gradient is
compared along the sky modes, which are independent per channel: the gains' gradient contracts the filtered
residual with the smooth functions of frequency that the filter removes, so it is a difference of the two
sides' FP64 filter builds."""
import numpy as np
import pytest

import oracle
from gpu_cases import rel_l2
from paper_2504_07090_gb300 import synth

pytestmark = pytest.mark.gpu
TAU, EPS = 250e-9, 1e-8
BOUNDS = {"fp64": (1e-7, 5e-7), "fp32": (1e-5, 2e-5)}


@pytest.mark.parametrize("nf", [1, 2, 3, 4, 5, 7, 8, 9, 12, 15, 16, 31, 63, 64, 65, 72, 100])
@pytest.mark.parametrize("prec", list(BOUNDS))
def test_filtered_gradient_at_channel_counts(nf, prec):
    import torch
    from paper_2504_07090_gb300 import fm
    p = synth.drift_scan_problem("filter", 2, nf, 140e6, 160e6, 3, 3, 8, 4, 2, 20, 5, ant_enu=synth.hex_array(2)[:5])
    p.sigma = 100.0
    th = synth.draw_truth(p).theta.astype(np.float32).astype(float)
    d = synth.random_data(p, 1e4, 6).astype(np.float32).astype(float)
    h = fm.ForwardModel(p, prec)
    h.set_data(torch.tensor(d, dtype=h.dtype, device="cuda").contiguous())
    h.set_delay_filter(TAU, EPS)
    scal, grad = h.chi2_grad(torch.tensor(th, dtype=h.dtype, device="cuda"))
    chi2, _, g = oracle.Oracle(p).chi2_grad_filtered(th, d[..., 0] + 1j * d[..., 1], oracle.delay_filter(p.freq_hz, TAU, EPS))
    b_c, b_g = BOUNDS[prec]
    if nf > 1:                       # one channel: the filter leaves 1e-8 of everything
        assert abs(float(scal[0]) - chi2) < b_c * chi2
        assert rel_l2(grad.cpu().numpy()[: p.n_sky_params], g[: p.n_sky_params]) < b_g
    h.sync_status()
    h.close()
