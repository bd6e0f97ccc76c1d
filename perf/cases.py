"""The calls that a user of this package makes, as measurable cases.

Each case is one pass through the public binding (``paper_2504_07090_gb300.fm``) on a seeded
drift scan: chi^2 gradients, Hessian-vector products, visibilities, sky maps, the mass-matrix
build, one iteration of the device chain and a batch of trajectories.  Sizes are those of the
named workloads (``synth.config``) and of what lies between them.

Inputs come from the seed and from the reference below, which states the model of
Eq. rime_discrete in 64 bits with torch alone; ``exact`` evaluates the same calls with it.
"""
import math

import numpy as np
import torch

from paper_2504_07090_gb300 import fm, synth

C_LIGHT = 299792458.0
TAU_MAX_S, NOISE_RATIO = 250e-9, 1e-8      # delay filter of the paper
N_STEPS, A_MIN = 20, 0.2                   # leapfrog steps of a trajectory, threshold of the step rule
ACCEPT_U = 0.01                            # accept uniform of the batched trajectories

SIZES = {
    # 7-antenna hexagon, 16 channels, 20 LSTs, 32 x 96 pixels, 512 modes a channel
    "cfg0": dict(side=2, n_freq=16, f_lo=150e6, f_hi=160e6, n_lst=20, n_dec=32, n_ra=96, n_mode_ra=32, n_mode_dec=16),
    # 37-antenna hexagon, 64 channels, 60 LSTs, 128 x 192 pixels, 16,384 modes a channel
    "cfg1": dict(side=4, n_freq=64, f_lo=140e6, f_hi=160e6, n_lst=60, n_dec=128, n_ra=192, n_mode_ra=128,
                 n_mode_dec=128),
    # 127-antenna hexagon, 128 channels, 120 LSTs, 256 x 384 pixels, 65,536 modes a channel
    "cfg4": dict(side=7, n_freq=128, f_lo=120e6, f_hi=180e6, n_lst=120, n_dec=256, n_ra=384, n_mode_ra=256,
                 n_mode_dec=256),
}


def _case(name, op, size, precision, **more):
    return {"name": name, "op": op, "precision": precision, **SIZES[size], **more}


def listed():
    return [
        # the plain FP64 run of the small array: chi^2 and gradient, complex128 throughout
        _case("cfg0_grad_fp64", "grad", "cfg0", "fp64"),
        # the smallest call: model visibilities of the small array, for simulation and plots
        _case("cfg0_vis_bf16x3", "vis", "cfg0", "bf16x3"),
        # sky maps of a sample's modes (posterior means and variances are taken over these)
        _case("cfg1_maps_fp16x3", "maps", "cfg1", "fp16x3"),
        # chi^2 gradient of the HERA-like array, the step of every optimiser and sampler
        _case("cfg1_grad_fp16x3", "grad", "cfg1", "fp16x3"),
        # the same with the delay filter of the likelihood
        _case("cfg1_filter_bf16x3", "grad", "cfg1", "bf16x3", delay_filter=True),
        # the same in plain FP32, for users who want no split products
        _case("cfg1_grad_fp32", "grad", "cfg1", "fp32"),
        # 5-minute integrations on a pixelisation of its own (the paper's mock): no drift-scan symmetry
        _case("offgrid_grad_bf16x3", "grad", "cfg1", "bf16x3", n_lst=12, n_ra=160),
        # Gauss-Newton Hessian-vector product: Newton steps and Laplace approximations take thousands
        _case("cfg1_hvp_fp16x3", "hvp", "cfg1", "fp16x3", full=False),
        # mass matrix of the sampler and a momentum drawn from it
        _case("cfg1_mass_fp16x3", "mass", "cfg1", "fp16x3"),
        # one iteration of the sampler on the device: momentum, 20 leapfrog steps, accept test
        _case("cfg1_chain_fp16x3", "chain", "cfg1", "fp16x3", eps=0.005),
        # trajectories of 16 independent chains of uneven size in one launch
        {"name": "cfg2_batch_bf16x3", "op": "batch", "precision": "bf16x3", "count": 16, "pick": 20250411},
        # chi^2 gradient of the largest array
        _case("cfg4_grad_fp16x3", "grad", "cfg4", "fp16x3"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    op = rng.choice(["grad", "grad", "grad", "vis", "hvp", "maps", "mass", "chain", "batch"])
    split = rng.choice(["fp16x3", "bf16x3", "fp16x3", "bf16x3", "fp16x1", "bf16x1"])
    if op == "batch":
        return {"op": op, "precision": split, "count": rng.randint(2, 12), "pick": rng.randint(1, 10 ** 6)}
    c = {"op": op, "precision": split, "side": rng.choice([2, 3, 4, 4, 5]), "n_freq": _log_int(rng, 3, 64)}
    c["f_lo"], c["f_hi"] = rng.choice([(140e6, 160e6), (150e6, 160e6), (120e6, 180e6)])
    if rng.random() < 0.3:                       # an array with antennas missing
        c["n_ant"] = rng.randint(3, 3 * c["side"] * (c["side"] - 1) + 1)
    if rng.random() < 0.65:                      # LST step of k / q pixels
        while True:
            m, (k, q) = rng.randint(1, 16), rng.choice([(1, 1), (1, 1), (2, 1), (3, 1), (1, 2), (3, 2), (3, 4)])
            if (16 * m * k) % q == 0 and 32 <= 16 * m * k // q <= 240:
                c["n_lst"], c["n_ra"] = 5 * m, 16 * m * k // q
                break
    else:
        c["n_lst"], c["n_ra"] = _log_int(rng, 2, 24), rng.randint(32, 240)
    c["n_dec"] = _log_int(rng, 12, 160)
    c["n_mode_ra"], c["n_mode_dec"] = 2 * _log_int(rng, 4, 64), _log_int(rng, 4, 128)
    if op in ("mass", "chain"):                  # 64 modes to a block
        c["n_mode_ra"], c["n_mode_dec"] = 16 * _log_int(rng, 1, 8), 4 * _log_int(rng, 1, 32)
    if op == "grad":
        if rng.random() < 0.35:
            c["precision"] = rng.choice(["fp32", "fp64"])
            n = (c.get("n_ant", 3 * c["side"] * (c["side"] - 1) + 1)) ** 2 / 2
            most = (3e10 if c["precision"] == "fp32" else 1e9) / (n * c["n_dec"] * c["n_ra"] * c["n_lst"])
            c["n_freq"] = max(1, min(c["n_freq"], int(most)))
        elif rng.random() < 0.3:
            c["delay_filter"] = True
        elif rng.random() < 0.4:
            c["n_freq_modes"] = rng.randint(1, min(6, c["n_freq"]))
        c["airy"] = rng.random() < 0.25
    if op == "hvp":
        c["full"] = rng.random() < 0.5
    if op == "chain":
        c["eps"] = 0.005
    return c


# ----------------------------------------------------------------------------- inputs

def _problem(c):
    p = synth.drift_scan_problem(c.get("name", "drawn"), c["side"], c["n_freq"], c["f_lo"], c["f_hi"], c["n_lst"],
                                 c["n_dec"], c["n_ra"], c["n_mode_ra"], c["n_mode_dec"])
    if "n_ant" in c:
        p.ant_enu = np.ascontiguousarray(p.ant_enu[: c["n_ant"]])
    if c.get("n_freq_modes"):
        p = synth.with_freq_modes(p, c["n_freq_modes"])
    return synth.with_airy_beam(p) if c.get("airy") else p


def _problems(c):
    return synth.batch_problems(c["count"], c["pick"]) if c["op"] == "batch" else [_problem(c)]


def _params(p, gen):
    """Sky modes (200 K of diffuse emission with 30 % fluctuations that fall off with wavenumber and
    degree as nu^-2.5, and a white part that differs from row to row) and gains 1 + 0.05 CN(0, 1)."""
    dev = torch.device("cuda")
    rows, M, N = p.n_sky_rows, p.n_mode_ra, p.n_mode_dec
    mean = float(synth.rayleigh_jeans_jy_per_sr(200.0, synth.NU0_HZ))
    k = (torch.arange(M, device=dev, dtype=torch.float64)[:, None] + 1.0).div(2, rounding_mode="floor")
    n = torch.arange(N, device=dev, dtype=torch.float64)[None, :]
    a = 0.3 * mean * ((1 + k) * (1 + n)) ** -1.5 * torch.randn(M, N, generator=gen, device=dev, dtype=torch.float64)
    if p.n_freq_modes:
        scale = 0.2 ** torch.arange(rows, device=dev, dtype=torch.float64)
    else:
        scale = torch.tensor((p.freq_hz / synth.NU0_HZ) ** -2.5, device=dev)
    white = 1e-3 * mean * torch.randn(rows, M, N, generator=gen, device=dev, dtype=torch.float64)
    sky = scale[:, None, None] * a + white
    sky[:, 0, 0] = (scale if not p.n_freq_modes else scale * (torch.arange(rows, device=dev) == 0)) * mean
    g = 0.05 / math.sqrt(2.0) * torch.randn(p.n_ant, p.n_gain, 2, generator=gen, device=dev, dtype=torch.float64)
    g[:, 0, 0] += 1.0
    return torch.cat([sky.reshape(-1), g.reshape(-1)])


def _prior(p, theta):
    """Widths of 5 % of each row's rms for the sky modes and of 0.05 for the gains."""
    sky = theta[: p.n_sky_params].reshape(p.n_sky_rows, -1)
    lam = torch.full_like(theta, 1.0 / 0.05 ** 2)
    lam[: p.n_sky_params] = (1.0 / (0.05 * sky.square().mean(1, keepdim=True).sqrt()) ** 2).expand_as(sky).reshape(-1)
    return theta.clone(), lam


def _inputs(p, c, seed):
    """What the calls get, in the precision they get it in."""
    dt = torch.float64 if c["precision"] == "fp64" else torch.float32
    gen = torch.Generator(device="cuda").manual_seed(1000003 * seed + p.seed % 1000003)

    def randn(*shape):
        return torch.randn(*shape, generator=gen, device="cuda", dtype=dt)

    truth = _params(p, gen)
    i = {"theta": truth.to(dt)}
    if c["op"] in ("vis", "maps"):
        return i
    ref = Reference(p)
    if c["op"] in ("mass", "chain", "batch"):
        # sampling: the data are the model of the truth and noise of 1 % of the mean visibility
        m = ref.model(ref.group_vis(i["theta"].double()), i["theta"].double())
        i["sigma"] = 0.01 * float(m.abs().mean())
        i["data"] = (torch.view_as_real(m) + i["sigma"] * randn(*m.shape, 2)).to(dt)
        i["z"] = randn(p.n_params)
    else:
        # the first steps of a fit: the data are of the model's size and know nothing of this sky
        m = ref.model(ref.group_vis(truth, [p.n_freq // 2]), truth, [p.n_freq // 2])
        rms = float(m.abs().square().mean().sqrt())
        i["sigma"] = 0.01 * rms
        i["data"] = randn(p.n_freq, p.n_lst, p.n_bl, 2).mul_(rms / math.sqrt(2.0))
        i["v"] = randn(p.n_params)
    mu, lam = _prior(p, truth)
    i["mu"], i["lam"] = mu.to(dt), lam.to(dt)
    return i


def _handle(p, c, i):
    h = fm.ForwardModel(p, c["precision"], sigma=i.get("sigma", 1.0))
    if "data" in i:
        h.set_data(i["data"])
        h.set_prior(i["mu"], i["lam"])
    if c.get("delay_filter"):
        h.set_delay_filter(TAU_MAX_S, NOISE_RATIO)
    return h


def _step(p):
    """Leapfrog step of a chain of the batch: 0.007 at 1.05e6 parameters, growing as n^(-1/4)."""
    return min(0.03, 0.007 * (1048872.0 / p.n_params) ** 0.25)


def prepare(case, seed):
    ps = _problems(case)
    ins = [_inputs(p, case, seed) for p in ps]
    hs = [_handle(p, case, i) for p, i in zip(ps, ins)]
    s = {"op": case["op"], "seed": seed, "case": case, "hs": hs, "h": hs[0], **ins[0]}
    if case["op"] in ("chain", "batch"):
        for h, i in zip(hs, ins):
            h.build_precond(i["theta"], 64)
    if case["op"] == "grad" and case["precision"] != "fp64":
        s["theta"].requires_grad_(True)
    if case["op"] == "chain":
        s["q"] = s["theta"].clone()
        s["start"] = torch.tensor([case["eps"], 0.0], dtype=torch.float64, device="cuda")
        s["state"] = s["start"].clone()
    if case["op"] == "batch":
        s["q0"], s["z"] = [i["theta"] for i in ins], [i["z"] for i in ins]
        s["q"], s["p"] = [q.clone() for q in s["q0"]], [torch.empty_like(q) for q in s["q0"]]
        s["batch"] = fm.Batch(hs, s["q"], s["p"], N_STEPS)
        s["eps"], s["u"] = [_step(p) for p in ps], [ACCEPT_U] * len(ps)
    return s


# ----------------------------------------------------------------------------- the calls

def run(s):
    h = s["h"]
    if s["op"] == "vis":
        return h.forward(s["theta"])
    if s["op"] == "maps":
        return h.sky_pixels(s["theta"])
    if s["op"] == "hvp":
        return h.hvp(s["theta"], s["v"], full=s["case"]["full"])
    if s["op"] == "mass":
        h.build_precond(s["theta"], 64)
        return h.precond_apply(0, s["z"])
    if s["op"] == "chain":
        s["q"].copy_(s["theta"])
        s["state"].copy_(s["start"])
        h.hmc_chain(s["q"], 1, N_STEPS, s["case"]["eps"], A_MIN, s["seed"], s["state"])
        return {"q": s["q"], "state": s["state"]}
    if s["op"] == "batch":
        torch._foreach_copy_(s["q"], s["q0"])
        for h, z, p in zip(s["hs"], s["z"], s["p"]):
            h.precond_apply(0, z, p)
        _, accepted = s["batch"].run(s["eps"], s["u"])
        return {"q": s["q"], "accepted": accepted}
    if s["case"]["precision"] == "fp64":
        scal, grad = h.chi2_grad(s["theta"])
        return {"chi2_u": scal, "grad": grad}
    s["theta"].grad = None
    u = fm.chi2_potential(s["theta"], h)
    u.backward()
    return {"u": u.detach(), "grad": s["theta"].grad}


# ----------------------------------------------------------------------------- work

def _groups(p):
    """Baselines that differ by more than their sign: (representatives, group of each, sign of each)."""
    i, j = np.triu_indices(p.n_ant, 1)
    b = np.round((p.ant_enu[i] - p.ant_enu[j]) * 1e6).astype(np.int64)
    first = np.where(b[:, 0] != 0, b[:, 0], np.where(b[:, 1] != 0, b[:, 1], b[:, 2]))
    sign = np.where(first < 0, -1, 1)
    _, rep, group = np.unique(b * sign[:, None], axis=0, return_index=True, return_inverse=True)
    return (p.ant_enu[i] - p.ant_enu[j])[rep] * sign[rep][:, None], group.reshape(-1), sign


def work(case):
    out = {"bytes": 0.0, "flops": 0.0}
    for p in _problems(case):
        U, ft = len(_groups(p)[0]), p.n_freq * p.n_lst
        real = 8 if case["precision"] == "fp64" else 4
        maps = 2.0 * p.n_freq * min(p.n_modes * p.n_dec + p.n_dec * p.n_mode_ra * p.n_ra,
                                    p.n_modes * p.n_ra + p.n_ra * p.n_mode_dec * p.n_dec)
        fringe = 4.0 * U * p.n_pix * ft                       # one sum over the pixels and its fringes
        grad, state, vis = 2 * (maps + fringe), real * p.n_params, 2 * real * p.n_vis
        if case["op"] == "maps":
            b, f = state + real * p.n_freq * p.n_pix, maps
        elif case["op"] == "vis":
            b, f = state + vis, maps + fringe
        elif case["op"] == "hvp":
            b, f = 4 * state + (vis if case["full"] else 0), 3 * (maps + fringe)
        elif case["op"] == "mass":
            gram = 2.0 * p.n_modes * 64 * 2 * U * ft
            per = p.n_modes * p.n_dec + p.n_dec * p.n_mode_ra * p.n_ra
            b, f = 4 * state, gram + 2.0 * 2 * U * ft * per
        elif case["op"] in ("chain", "batch"):
            b, f = 5 * state + vis + real * 64 * p.n_params, (N_STEPS + 1) * grad
        else:
            b, f = 4 * state + vis, grad
        out = {"bytes": out["bytes"] + b, "flops": out["flops"] + f}
    return out


# ----------------------------------------------------------------------------- the reference in 64 bits

class Reference:
    """The model and its derivatives in FP64: one channel at a time, the response of every distinct
    baseline over the distinct hour angles as one matrix."""

    def __init__(self, p):
        f64 = dict(dtype=torch.float64, device="cuda")
        self.p = p
        vec, group, sign = _groups(p)
        self.vec, self.U = torch.tensor(vec, **f64), len(vec)
        self.group = torch.tensor(group, device="cuda")
        self.sign = torch.tensor(sign, **f64)
        i, j = np.triu_indices(p.n_ant, 1)
        self.i, self.j = torch.tensor(i, device="cuda"), torch.tensor(j, device="cuda")
        dra, ddec = (p.ra_max - p.ra_min) / p.n_ra, (p.dec_max - p.dec_min) / p.n_dec
        ra = p.ra_min + (np.arange(p.n_ra) + 0.5) * dra
        edge = p.dec_min + np.arange(p.n_dec + 1) * ddec
        dec = 0.5 * (edge[1:] + edge[:-1])
        H = p.lst_rad[:, None] - ra[None, :]
        _, at, cell = np.unique(np.round(H * 1e9), return_index=True, return_inverse=True)
        self.cell = torch.tensor(cell.reshape(H.shape), device="cuda")          # [T][R]
        self.n_cell = len(at)
        h, d = H.reshape(-1)[at][None, :], dec[:, None]
        sl, cl = math.sin(p.lat_rad), math.cos(p.lat_rad)
        s = np.stack([-np.cos(d) * np.sin(h), cl * np.sin(d) - sl * np.cos(d) * np.cos(h),
                      sl * np.sin(d) + cl * np.cos(d) * np.cos(h)])
        self.s = torch.tensor(s, **f64)                                         # [3][D][cells]
        self.domega = torch.tensor(dra * np.diff(np.sin(edge)), **f64)
        ahat = 2 * np.pi * (ra - p.ra_min) / (p.ra_max - p.ra_min)
        M = p.n_mode_ra
        phi = [np.ones_like(ahat)] + [np.cos((m + 1) // 2 * ahat) if m % 2 else np.sin(m // 2 * ahat)
                                      for m in range(1, M - 1)] + [np.cos(0.5 * M * ahat)]
        self.phi = torch.tensor(np.stack(phi, 1), **f64)
        x = 2 * (dec - p.dec_min) / (p.dec_max - p.dec_min) - 1
        self.leg = torch.tensor(np.polynomial.legendre.legvander(x, p.n_mode_dec - 1), **f64)
        span = p.freq_hz[-1] - p.freq_hz[0]
        nu = 2 * (p.freq_hz - p.freq_hz[0]) / span - 1 if span > 0 else np.zeros(p.n_freq)
        self.gleg = torch.tensor(np.polynomial.legendre.legvander(nu, p.n_gain - 1), **f64)
        self.fleg = torch.tensor(np.polynomial.legendre.legvander(nu, max(p.n_freq_modes, 1) - 1), **f64)
        self.kept = {}

    def response(self, f):
        """[2 U][D][cells]: solid angle times beam times the real and imaginary parts of the fringe."""
        if f in self.kept:
            return self.kept[f]
        p, nu = self.p, float(self.p.freq_hz[f])
        up = self.s[2]
        if p.beam_type:
            e, n = self.s[0], self.s[1]
            x = (p.dish_ns_m * n * n + p.dish_ew_m * e * e) / (e * e + n * n).sqrt().clamp_min(1e-300) * math.pi * nu / C_LIGHT
            beam = torch.where(x > 1e-7, 2 * torch.special.bessel_j1(x) / x.clamp_min(1e-300), torch.ones_like(x)) ** 2
        else:
            fwhm = p.beam_fwhm_ref_rad * p.beam_ref_hz / nu
            beam = torch.exp(-4 * math.log(2.0) * torch.atan2((self.s[0] ** 2 + self.s[1] ** 2).sqrt(), up) ** 2 / fwhm ** 2)
        w = torch.where(up > 0, beam, torch.zeros_like(beam)) * self.domega[:, None]
        turns = torch.tensordot(self.vec * (nu / C_LIGHT), self.s, 1)
        turns = 2 * math.pi * (turns - turns.round())
        P = torch.cat([w * torch.cos(turns), -w * torch.sin(turns)])
        if P.numel() * 8 * p.n_freq < 8e9:
            self.kept[f] = P
        return P

    def modes(self, theta):
        a = theta[: self.p.n_sky_params].reshape(self.p.n_sky_rows, -1)
        a = self.fleg @ a if self.p.n_freq_modes else a
        return a.reshape(self.p.n_freq, self.p.n_mode_ra, self.p.n_mode_dec)

    def gamma(self, theta):
        return theta[self.p.n_sky_params:].reshape(self.p.n_ant, self.p.n_gain, 2)

    def pixels(self, theta):
        return self.leg @ self.modes(theta).transpose(1, 2) @ self.phi.T           # [F][D][R]

    def group_vis(self, theta, channels=None):
        """[F][T][2][U]: the distinct visibilities of the sky modes in theta."""
        p, x, out = self.p, self.pixels(theta), []
        at = self.cell[:, None, :].expand(-1, p.n_dec, -1)
        for f in range(p.n_freq) if channels is None else channels:
            X = torch.zeros(p.n_lst, p.n_dec, self.n_cell, dtype=torch.float64, device="cuda")
            X.scatter_(2, at, x[f].expand(p.n_lst, -1, -1))
            out.append((X.reshape(p.n_lst, -1) @ self.response(f).reshape(2 * self.U, -1).T).reshape(-1, 2, self.U))
        return torch.stack(out)

    def modes_back(self, q):
        """Transpose of group_vis: [F][T][2][U] to the sky parameters."""
        p, out = self.p, []
        at = self.cell[:, None, :].expand(-1, p.n_dec, -1)
        for f in range(p.n_freq):
            X = (q[f].reshape(p.n_lst, -1) @ self.response(f).reshape(2 * self.U, -1)).reshape(p.n_lst, p.n_dec, -1)
            out.append((self.leg.T @ X.gather(2, at).sum(0) @ self.phi).T.reshape(-1))
        a = torch.stack(out)
        return (self.fleg.T @ a if p.n_freq_modes else a).reshape(-1)

    def _model(self, v, gamma, channels=None):
        g = torch.einsum("fk,akc->fac", self.gleg if channels is None else self.gleg[channels], gamma)
        g = torch.complex(g[..., 0], g[..., 1])
        V = torch.complex(v[:, :, 0][..., self.group], self.sign * v[:, :, 1][..., self.group])
        return (g[:, self.i] * g[:, self.j].conj())[:, None, :] * V

    def model(self, v, theta, channels=None):
        return self._model(v, self.gamma(theta), channels)

    def delay_filter(self):
        nu = torch.tensor(self.p.freq_hz, dtype=torch.float64, device="cuda")
        fg = torch.sinc(2 * TAU_MAX_S * (nu[:, None] - nu[None, :]))
        eye = torch.eye(len(nu), dtype=torch.float64, device="cuda")
        # C_fg and C_noise = e I commute: I - C_fg (C_fg + e I)^-1 = e (C_fg + e I)^-1
        return NOISE_RATIO * torch.linalg.inv(fg + NOISE_RATIO * eye)

    def grad(self, theta, i, filtered=False):
        """(chi^2, U, gradient of U)"""
        data = torch.view_as_complex(i["data"].double())
        with torch.enable_grad():
            v = self.group_vis(theta).requires_grad_(True)
            gamma = self.gamma(theta).clone().requires_grad_(True)
            r = self._model(v, gamma) - data
            if filtered:
                F = self.delay_filter()
                r = torch.einsum("fg,gtb->ftb", F.to(r.dtype), r) / F.square().sum(1).sqrt()[:, None, None]
            chi2 = (r.real.square() + r.imag.square()).sum() / i["sigma"] ** 2
            gv, gg = torch.autograd.grad(0.5 * chi2, (v, gamma))
        off = theta - i["mu"].double()
        lam = i["lam"].double()
        u = 0.5 * chi2.detach() + 0.5 * (lam * off * off).sum()
        return chi2.detach(), u, torch.cat([self.modes_back(gv), gg.reshape(-1)]) + lam * off

    def hvp(self, theta, i, full):
        data, vec = torch.view_as_complex(i["data"].double()), i["v"].double()
        at = (self.group_vis(theta), self.gamma(theta))
        along = (self.group_vis(vec), self.gamma(vec))
        if full:
            def u(v, gamma):
                return 0.5 * torch.view_as_real(self._model(v, gamma) - data).square().sum() / i["sigma"] ** 2
            hv, hg = torch.func.jvp(torch.func.grad(u, argnums=(0, 1)), at, along)[1]
        else:
            def m(v, gamma):
                return torch.view_as_real(self._model(v, gamma))
            dm = torch.func.jvp(m, at, along)[1]
            hv, hg = torch.func.vjp(m, *at)[1](dm / i["sigma"] ** 2)
        return torch.cat([self.modes_back(hv), hg.reshape(-1)]) + i["lam"].double() * vec

    def mass(self, theta, i):
        """Cholesky factors of the Gauss-Newton mass matrix: [sky blocks][64][64] and the gain block."""
        p, U = self.p, self.U
        V, gamma = self.group_vis(theta), self.gamma(theta)
        g = torch.einsum("fk,akc->fac", self.gleg, gamma)
        g = torch.complex(g[..., 0], g[..., 1])
        gg = (g[:, self.i] * g[:, self.j].conj()).abs().square()
        W = torch.zeros(p.n_freq, U, dtype=torch.float64, device="cuda").index_add_(1, self.group, gg)
        nb = p.n_modes // 64
        sky = []
        for f in range(p.n_freq):
            G, P, w = 0, self.response(f), W[f].repeat(2)[None, :, None]
            for t in range(p.n_lst):
                C = (P[:, :, self.cell[t]] @ self.phi).transpose(1, 2) @ self.leg       # [2U][M][N]
                C = C.reshape(2 * U, nb, 64).transpose(0, 1)
                G = G + (C * w).transpose(1, 2) @ C
            sky.append(G)
        sky = torch.cat(sky) / i["sigma"] ** 2
        ng = p.n_ant * p.n_gain * 2
        gain = torch.zeros(p.n_ant, p.n_gain, 2, p.n_ant, p.n_gain, 2, dtype=torch.float64, device="cuda")
        Vb = torch.complex(V[:, :, 0][..., self.group], self.sign * V[:, :, 1][..., self.group])
        row = torch.arange(p.n_bl, device="cuda")
        for f in range(p.n_freq):
            J = torch.zeros(p.n_lst, p.n_bl, p.n_ant, 2, dtype=torch.complex128, device="cuda")
            ci, cj = g[f, self.j].conj() * Vb[f], g[f, self.i] * Vb[f]
            J[:, row, self.i, 0], J[:, row, self.i, 1] = ci, 1j * ci
            J[:, row, self.j, 0], J[:, row, self.j, 1] = cj, -1j * cj
            J = torch.view_as_real(J.reshape(-1, 2 * p.n_ant)).permute(0, 2, 1).reshape(-1, 2 * p.n_ant)
            JJ = (J.T @ J).reshape(p.n_ant, 2, p.n_ant, 2) / i["sigma"] ** 2
            gain += torch.einsum("acbd,k,l->akcbld", JJ, self.gleg[f], self.gleg[f])
        lam = i["lam"].double()
        sky = sky + torch.diag_embed(lam[: p.n_sky_params].reshape(-1, 64))
        gain = gain.reshape(ng, ng) + torch.diag(lam[p.n_sky_params:])
        return torch.linalg.cholesky(sky), torch.linalg.cholesky(gain)

    def times_factor(self, L, z):
        n = self.p.n_sky_params
        return torch.cat([(L[0] @ z[:n].reshape(-1, 64, 1)).reshape(-1), L[1] @ z[n:]])

    def solve(self, L, p):
        n = self.p.n_sky_params
        return torch.cat([torch.cholesky_solve(p[:n].reshape(-1, 64, 1), L[0]).reshape(-1),
                          torch.cholesky_solve(p[n:, None], L[1]).reshape(-1)])

    def trajectory(self, i, eps):
        """Final position of a leapfrog trajectory and whether it is accepted."""
        q = i["theta"].double()
        L = self.mass(q, i)
        p = self.times_factor(L, i["z"].double())
        _, u0, g = self.grad(q, i)
        h0 = u0 + 0.5 * i["z"].double().square().sum()
        for _ in range(N_STEPS):
            p = p - 0.5 * eps * g
            q = q + eps * self.solve(L, p)
            _, u, g = self.grad(q, i)
            p = p - 0.5 * eps * g
        h1 = u + 0.5 * (p * self.solve(L, p)).sum()
        accepted = bool(torch.exp(h0 - h1) > ACCEPT_U)
        return (q if accepted else i["theta"].double()), torch.tensor([int(accepted)], dtype=torch.int32, device="cuda")


def exact(case, seed):
    ps = _problems(case)
    if case["op"] == "chain":
        return None              # its momenta come from the package's own generator
    if case["op"] == "batch":
        got = [Reference(p).trajectory(_inputs(p, case, seed), _step(p)) for p in ps]
        return {"q": [q for q, _ in got], "accepted": [a for _, a in got]}
    p, i = ps[0], _inputs(ps[0], case, seed)
    ref, theta = Reference(p), i["theta"].double()
    if case["op"] == "vis":
        return torch.view_as_real(ref.model(ref.group_vis(theta), theta))
    if case["op"] == "maps":
        return ref.pixels(theta).reshape(-1)
    if case["op"] == "hvp":
        return ref.hvp(theta, i, case["full"])
    if case["op"] == "mass":
        return ref.times_factor(ref.mass(theta, i), i["z"].double())
    chi2, u, g = ref.grad(theta, i, bool(case.get("delay_filter")))
    if case["precision"] == "fp64":
        return {"chi2_u": torch.stack([chi2, u]), "grad": g}
    return {"u": u, "grad": g}
