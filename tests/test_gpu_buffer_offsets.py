"""Caller's buffers that start one element into an allocation (aligned for a real, not for a complex pair or a
16-byte word): every contraction form reads and writes them with the same results, bit for bit, as aligned ones."""
import numpy as np
import pytest

from paper_2504_07090_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("airy", [False, True])
@pytest.mark.parametrize("grid", ["drift", "offgrid"])
@pytest.mark.parametrize("prec", ["fp64", "fp32", "fp16x3", "bf16x1"])
def test_offset_buffers_give_the_same_bits(prec, grid, airy):
    import torch
    from paper_2504_07090_gb300 import fm
    p = synth.drift_scan_problem("offset", 3, 3, 150e6, 155e6, 5, 5, 32 if grid == "drift" else 29, 16, 4, 20, 19)
    h = fm.ForwardModel(synth.with_airy_beam(p) if airy else p, prec, sigma=1.0)

    def put(a, off):
        buf = torch.zeros(a.size + 3, dtype=h.dtype, device="cuda")
        buf[off:off + a.size] = torch.tensor(np.ascontiguousarray(a).reshape(-1), device="cuda").to(h.dtype)
        return buf[off:off + a.size]

    tr = synth.draw_truth(p)
    x = np.random.default_rng(2).standard_normal(h.n_pix_total)
    v = synth.random_vectors(h.n_params, 1, 4)[0]
    got = []
    for off in (0, 1):
        th, xx, vv = put(tr.theta, off), put(x, off), put(v, off)
        vis, visx, grad, hv = (put(np.zeros(n), off) for n in (2 * h.n_vis, 2 * h.n_vis, h.n_params, h.n_params))
        assert vis.data_ptr() % (2 * vis.element_size()) == off * vis.element_size()
        h.set_data(put(synth.random_data(p, 1e4, 3), off))
        h.forward(th, vis)
        h.forward_pixels(xx, visx)
        scal, _ = h.chi2_grad(th, grad)
        h.hvp(th, vv, out=hv)
        got.append([t.clone() for t in (vis, visx, grad, hv, scal)])
    h.sync_status()
    h.close()
    for a, b in zip(*got):
        assert torch.equal(a, b) and float(a.abs().max()) > 0
