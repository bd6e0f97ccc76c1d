"""FP32 handles of large arrays without redundancy (every baseline a fringe of its own) in hour-angle modes against the
per-baseline sums: gradients up to the largest array whose per-baseline epilogue fits a CTA (138 antennas), and
Hessian-vector products from where a baseline list passes 48 KB (111 antennas) to the largest that the tangent
epilogue takes (120).  Bounds: those of the large-array epilogue (chi^2 2e-5, gradients and products 1e-4)."""
import numpy as np
import pytest

from paper_2504_07090_gb300 import synth

pytestmark = pytest.mark.gpu


def _problem(n_ant):
    ant = synth.hex_array(8)[:n_ant] + 0.5 * np.random.default_rng(7).standard_normal((n_ant, 3)) * [1.0, 1.0, 0.1]
    return synth.drift_scan_problem("random", 7, 2, 150e6, 153e6, 3, 3, 32, 8, 4, 20, 41, ant_enu=ant)


def _both(p, monkeypatch, call):
    import torch
    from paper_2504_07090_gb300 import fm
    th = torch.tensor(synth.draw_truth(p).theta.astype(np.float32), device="cuda")
    d = torch.tensor(synth.random_data(p, 1e4, 3).astype(np.float32), device="cuda")
    out = []
    for ha in ("1", "0"):
        monkeypatch.setenv("FM_HA", ha)
        h = fm.ForwardModel(p, "fp32", sigma=1.0)
        assert (h.mode_table_bytes() > 0) == (ha == "1")
        h.set_data(d)
        out.append(call(h, th))
        h.sync_status()
        h.close()
    return out


def _err(a, b):
    return float((a.double() - b.double()).norm() / b.double().norm())


@pytest.mark.parametrize("n_ant", [120, 121, 138])
def test_gradient_matches_per_baseline_sums(n_ant, monkeypatch):
    def call(h, th):
        scal, grad = h.chi2_grad(th)
        return float(scal[0]), grad.clone()
    (ca, ga), (cb, gb) = _both(_problem(n_ant), monkeypatch, call)
    assert abs(ca - cb) < 2e-5 * cb
    assert _err(ga, gb) < 1e-4


@pytest.mark.parametrize("n_ant", [110, 111, 120])
@pytest.mark.parametrize("full", [True, False])
def test_hessian_vector_product_matches_per_baseline_sums(n_ant, full, monkeypatch):
    import torch
    p = _problem(n_ant)
    v = torch.tensor(synth.random_vectors(p.n_params, 1, 4)[0].astype(np.float32), device="cuda")
    a, b = _both(p, monkeypatch, lambda h, th: h.hvp(th, v, full=full))
    assert _err(a, b) < 1e-4
