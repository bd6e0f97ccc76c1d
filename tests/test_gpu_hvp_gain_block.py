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


# channels and LSTs around the 64 and 64 that a pass of the sum takes; gain coefficients 1, past 8, the most
@pytest.mark.parametrize("nf,nt,ng", [(1, 1, 1), (3, 70, 9), (65, 2, 4), (130, 5, 16), (64, 64, 4), (2, 129, 1)])
@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_gain_block_is_the_sum_over_single_channels(nf, nt, ng, prec, monkeypatch):
    """With gains and directions flat in frequency the terms of a channel are those of a handle of that channel with one
    coefficient, weighted by the Legendre polynomials P_k.  FP64: rounding only.  FP32: the terms, the
    polynomials and the result are rounded to 2^-24 each."""
    import copy
    import torch
    from paper_2504_07090_gb300 import fm
    for k in ("FM_HA", "FM_HA_GROUPS"):
        monkeypatch.setenv(k, "0")
    p = synth.drift_scan_problem("gains", 2, nf, 150e6, 160e6, nt, 3, 16, 4, 4, 20, 41, n_gain=ng)
    f32 = lambda a: np.asarray(a).astype(np.float32).astype(np.float64)  # noqa: E731
    th, v = f32(synth.draw_truth(p).theta), f32(synth.random_vectors(p.n_params, 1, 4)[0])
    for x in (th, v):
        x[p.n_sky_params:].reshape(p.n_ant, ng, 2)[:, 1:] = 0.0
    d = f32(synth.random_data(p, 1e4, 3))

    def gains(q, theta, vec, data):
        h = fm.ForwardModel(q, prec, sigma=1.0)
        put = lambda a: torch.tensor(np.ascontiguousarray(a), device="cuda").to(h.dtype)  # noqa: E731
        h.set_data(put(data))
        out = h.hvp(put(theta), put(vec), full=True)[q.n_sky_params:].cpu().double().numpy()
        h.sync_status()
        h.close()
        return out.reshape(q.n_ant, q.n_gain, 2)

    got = gains(p, th, v, d)
    terms, nk = [], p.n_modes
    for f in range(nf):
        q = copy.copy(p)
        q.freq_hz, q.n_gain = p.freq_hz[f:f + 1].copy(), 1
        one = [np.concatenate([x[f * nk:(f + 1) * nk], x[p.n_sky_params:].reshape(p.n_ant, ng, 2)[:, 0].reshape(-1)])
               for x in (th, v)]
        terms.append(gains(q, *one, d[f:f + 1])[:, 0])
    x = 2 * (p.freq_hz - p.freq_hz[0]) / (p.freq_hz[-1] - p.freq_hz[0]) - 1 if nf > 1 else np.zeros(1)
    P = np.polynomial.legendre.legvander(x, ng - 1)
    want = np.einsum("fk,fac->akc", P, terms)
    size = np.einsum("fk,fac->akc", np.abs(P), np.abs(terms))
    slack = 1e-12 * size if prec == "fp64" else 2.0 ** -24 * (np.abs(want) + 2.1 * size)
    assert np.all(np.abs(got - want) <= slack), np.max(np.abs(got - want) / slack)
