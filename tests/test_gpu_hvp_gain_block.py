"""The gain block of a Hessian-vector product is summed over channels and LSTs in FP64.  With one channel and one gain
coefficient it is the plain sum of the per-LST terms, and handles of one LST each return those terms: in the
per-baseline form a term's arithmetic is the same in both, so the sum may differ by the rounding of its result
to FP32 only (2^-24 of it), whatever cancels."""
import numpy as np
import pytest

from paper_2504_07090_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("full", [True, False])
def test_gain_block_is_summed_in_fp64(full, monkeypatch):
    import copy
    import torch
    from paper_2504_07090_gb300 import fm
    for k in ("FM_HA", "FM_HA_GROUPS"):
        monkeypatch.setenv(k, "0")
    p = synth.drift_scan_problem("gain", 3, 1, 150e6, 150e6, 70, 5, 24, 8, 4, 20, 41, n_gain=1)
    th = torch.tensor(synth.draw_truth(p).theta.astype(np.float32), device="cuda")
    v = torch.tensor(synth.random_vectors(p.n_params, 1, 4)[0].astype(np.float32), device="cuda")
    d = torch.tensor(synth.random_data(p, 1e4, 3).astype(np.float32), device="cuda")

    def gains(q, data):
        h = fm.ForwardModel(q, "fp32", sigma=1.0)
        h.set_data(data.contiguous())
        out = h.hvp(th, v, full=full)[q.n_sky_params:].cpu().double().numpy()
        h.sync_status()
        h.close()
        return out

    got = gains(p, d)
    terms = []
    for t in range(p.n_lst):
        q = copy.copy(p)
        q.lst_rad = p.lst_rad[t:t + 1].copy()
        terms.append(gains(q, d[:, t:t + 1]))
    want = np.sum(terms, axis=0)
    slack = 2.0 ** -24 * np.abs(want) * (1 + 1e-6) + 1e-14 * np.sum(np.abs(terms), axis=0)
    assert np.all(np.abs(got - want) <= slack), np.max(np.abs(got - want) / slack)
