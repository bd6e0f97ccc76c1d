"""The CUDA-core mode -> pixel transform in FP32 at the edges of its 64 x 64 x 16 tiles, and its transpose in the
gradient, against FP64.

Bounds: FP32 sums of at most 130 terms, twice: 130 eps = 8e-6 at worst, 2e-6 in the l2 norm of sums of random
sign; the gradient adds the FP32 form's own (5e-5)."""
import numpy as np
import pytest

from paper_2504_07090_gb300 import synth

pytestmark = pytest.mark.gpu


# Dec and RA cells, RA and Dec modes
@pytest.mark.parametrize("nd, nr, mr, md", [(1, 8, 2, 1), (63, 64, 16, 15), (64, 65, 18, 16), (65, 63, 16, 17), (5, 130, 130, 3),
                                            (3, 129, 4, 130), (128, 16, 64, 65)])
def test_fp32_mode_transforms_match_fp64(nd, nr, mr, md):
    import torch
    from paper_2504_07090_gb300 import fm
    p = synth.drift_scan_problem("modes", 2, 2, 148e6, 152e6, 3, nd, nr, mr, md, 20, 3)
    th = np.random.default_rng(1).standard_normal(p.n_params).astype(np.float32)
    d = synth.random_data(p, 1e4, 3).astype(np.float32)
    out = {}
    for prec in ("fp32", "fp64"):
        h = fm.ForwardModel(p, prec, sigma=1.0)
        t = torch.tensor(th, device="cuda").to(h.dtype)
        h.set_data(torch.tensor(d, device="cuda").to(h.dtype))
        out[prec] = [h.sky_pixels(t).cpu().double(), h.chi2_grad(t)[1].cpu().double()]
        h.sync_status()
        h.close()
    for a, b, bound in zip(out["fp32"], out["fp64"], (2e-6, 5e-5)):
        assert float((a - b).norm() / b.norm()) < bound
