"""What the speed of the library is measured on.

Every case is a call that a user's program makes through the public Python
binding of libswig (``paper_2607_28265_gb300.swig``): batched likelihoods from
one parameter vector to several thousand, on host arrays, on device pointers
and on the allocation-free entry point; the full frequency grid in mixed and
FP64 precision, with phi_c or d_L marginalised; the heterodyned likelihood with
t_c sampled or marginalised; nested-sampling runs (their first iterations, from
the prior draws on); and the retraining of the learned proposal.  Sizes are
those of the repository's workloads (4 s and 32/64/128/256 s segments, H1/L1/V1,
20-2048 Hz, nlive 1000, 5,000 heterodyned bins, 2,000 time nodes), with odd
ones between them.

An event is made from a seed alone: an injection drawn from the prior, scaled
to a network SNR of 25, in Gaussian noise.  Parameter vectors are half drawn
from the prior (as a run starts) and half around the injection (as it ends).
``exact`` restates each likelihood in FP64 with torch.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2607_28265_gb300 import swig, workloads

si = workloads.si

NETWORK = ("H1", "L1", "V1")
SNR = 25.0


# ---------------------------------------------------------------------------
# Cases
# ---------------------------------------------------------------------------
def _loglike(name, seconds, dets, n, api="dev", marg="phase", f_max=2048.0):
    return {"name": name, "kind": "full", "seconds": seconds, "dets": dets, "f_max": f_max, "n": n, "api": api,
            "marg": marg}


def listed():
    return [
        # an outer program (another sampler, an optimiser) asks for one value at a time
        _loglike("one_theta_128s", 128, 3, 1, api="host"),
        # one evaluation of each chain of a run (nrep 100)
        _loglike("chains_128s", 128, 3, 100),
        # a live set (nlive 1000): a run's first step, a reweighting
        _loglike("live_set_128s", 128, 3, 1000),
        # a long segment and a batch over the library's internal split of 4096
        _loglike("wide_batch_256s", 256, 3, 4099),
        # a latency-critical loop that may not allocate: short segment, two detectors
        _loglike("noalloc_32s", 32, 2, 37, api="noalloc"),
        # d_L marginalised by quadrature
        _loglike("distance_marg_64s", 64, 3, 200, marg="distance"),
        # the 4 s single-detector FP64 reference configuration
        {"name": "fp64_4s", "kind": "fp64", "seconds": 4, "dets": 1, "f_max": 1024.0, "n": 100, "api": "dev",
         "marg": "none"},
        # the heterodyned likelihood over a live set
        {"name": "het_128s", "kind": "het", "seconds": 128, "dets": 3, "f_max": 2048.0, "n": 1000, "api": "dev",
         "marg": "phase", "bins": 5000, "spacing": 0},
        # ... with t_c marginalised on 2,000 nodes (the post-hoc pass over a run's samples)
        {"name": "het_time_marg_128s", "kind": "het", "seconds": 128, "dets": 3, "f_max": 2048.0, "n": 300,
         "api": "dev", "marg": "time", "bins": 5000, "spacing": 0, "nodes": 2000},
        # a posterior's first iterations on the full grid, samples read back
        {"name": "posterior_128s", "kind": "run", "seconds": 128, "dets": 3, "f_max": 2048.0, "nlive": 1000,
         "iters": 4, "bins": 0},
        # the same with the heterodyned likelihood
        {"name": "posterior_het_128s", "kind": "run", "seconds": 128, "dets": 3, "f_max": 2048.0, "nlive": 1000,
         "iters": 8, "bins": 5000},
        # one retraining of the learned proposal on a live set
        {"name": "retrain_1000", "kind": "retrain", "n": 1000, "d": 12, "steps": 30},
    ]


def _logint(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["full", "full", "full", "fp64", "het", "het", "run", "retrain"])
    seconds = _logint(rng, 32, 256)
    dets = rng.choice([2, 3]) if seconds < 64 else rng.choice([1, 2, 3])
    f_max = rng.choice([1024.0, 1500.0, 2048.0]) if seconds >= 64 else 2048.0
    if kind == "full":
        api = rng.choice(["dev", "dev", "host", "noalloc"])
        return {"kind": kind, "seconds": seconds, "dets": dets, "f_max": f_max,
                "n": _logint(rng, 1, 100 if api == "noalloc" else 4099), "api": api,
                "marg": rng.choice(["phase", "phase", "none", "distance"])}
    if kind == "fp64":
        return {"kind": kind, "seconds": rng.choice([4, 5, 8]), "dets": rng.choice([1, 2]), "f_max": 1024.0,
                "n": _logint(rng, 1, 300), "api": rng.choice(["dev", "host"]), "marg": rng.choice(["none", "phase"])}
    if kind == "het":
        c = {"kind": kind, "seconds": max(64, min(128, seconds)), "dets": rng.choice([2, 3]), "f_max": 2048.0,
             "n": _logint(rng, 1, 1000), "api": "dev", "marg": rng.choice(["phase", "phase", "none", "time"]),
             "bins": _logint(rng, 500, 5000), "spacing": rng.choice([0, 0, 1])}
        if c["marg"] == "time":
            c["n"] = min(c["n"], 300)
            c["nodes"] = _logint(rng, 64, 2000)
        return c
    if kind == "run":
        return {"kind": kind, "seconds": max(64, min(128, seconds)), "dets": rng.choice([2, 3]), "f_max": 2048.0,
                "nlive": _logint(rng, 200, 1000), "iters": rng.choice([1, 2, 3]),
                "bins": rng.choice([0, 0, _logint(rng, 1000, 5000)])}
    return {"kind": kind, "n": _logint(rng, 200, 1000), "d": rng.choice([4, 9, 12]), "steps": rng.randint(5, 30)}


# ---------------------------------------------------------------------------
# Events
# ---------------------------------------------------------------------------
def _params(case):
    """The prior: Table I of the workload, phi_c sampled, phi_c or d_L
    marginalised, or t_c marginalised; the 4 s configuration has its own."""
    if case["kind"] == "fp64":
        p = list(si.config1().params)
        if case["marg"] == "phase":
            p[12] = si.Param(si.PRIOR_UNIFORM, 0.0, 2 * math.pi, si.MODE_MARG)
        return p
    p = list(si.config2().params)
    marg = case.get("marg", "phase")
    if marg == "none":
        p[12] = si.Param(si.PRIOR_UNIFORM, 0.0, 2 * math.pi, block=8)
    if marg == "distance":
        p[6] = si.Param(p[6].kind, p[6].lo, p[6].hi, si.MODE_MARG)
    if marg == "time":
        p[11] = si.Param(p[11].kind, p[11].lo, p[11].hi, si.MODE_MARG)
    return p


def _draws(params, rng, n):
    """n parameter vectors from the prior (marginalised slots: any value in range)."""
    u = rng.random((n, si.N_PARAMS))
    th = np.empty((n, si.N_PARAMS))
    for j, p in enumerate(params):
        lo, hi = p.lo, p.hi
        if p.mode == si.MODE_FIXED:
            th[:, j] = p.value
        elif p.kind == si.PRIOR_SINE:
            th[:, j] = np.arccos(math.cos(lo) - u[:, j] * (math.cos(lo) - math.cos(hi)))
        elif p.kind == si.PRIOR_COSINE:
            th[:, j] = np.arcsin(math.sin(lo) + u[:, j] * (math.sin(hi) - math.sin(lo)))
        elif p.kind == si.PRIOR_POWER2:
            th[:, j] = np.cbrt(lo**3 + u[:, j] * (hi**3 - lo**3))
        else:
            th[:, j] = lo + u[:, j] * (hi - lo)
    return th


def _near(params, th, rng, n):
    """n parameter vectors around th: Mc and t_c by about their posterior
    widths, the others by a few percent of their ranges, inside the prior."""
    step = np.array([2e-4 * th[0], 0.01, 0.005, 0.005, 50.0, 50.0, 0.03 * th[6], 0.03, 0.05, 0.005, 0.005, 3e-4, 0.2])
    out = th + step * rng.standard_normal((n, si.N_PARAMS))
    for j, p in enumerate(params):
        out[:, j] = p.value if p.mode == si.MODE_FIXED else np.clip(out[:, j], p.lo, p.hi)
    return out


class _Event:
    """Grid, detectors, PSDs, prior and data of a case, in FP64 on the GPU."""

    def __init__(self, case, seed):
        rng = np.random.default_rng([seed, 17])
        self.case = case
        self.params = _params(case)
        self.f_min, self.f_max, self.df = 20.0, case["f_max"], 1.0 / case["seconds"]
        self.names = NETWORK[:case["dets"]]
        self.freqs = si.frequency_grid(self.f_min, self.f_max, self.df)
        self.f = torch.from_numpy(self.freqs).cuda()
        self.psds = [si.design_psd(self.freqs, si.PSD_SCALE[d]) for d in self.names]
        self.S = torch.from_numpy(np.stack(self.psds)).cuda()
        self.sites = [si.site_vectors(d) for d in self.names]
        self.gmst = si.gmst_from_gps(si.REFERENCE_GPS)
        th = si.config1().injection.copy() if case["kind"] == "fp64" else _draws(self.params, rng, 1)[0]
        h = self.strain(th)
        th[6] *= math.sqrt(float((4.0 * self.df * h.abs() ** 2 / self.S).sum())) / SNR
        self.theta0 = th
        gen = torch.Generator(device="cuda").manual_seed(int(seed) * 2 + 1)
        noise = torch.randn(2, *self.S.shape, generator=gen, device="cuda", dtype=torch.float64)
        self.data = self.strain(th) + torch.sqrt(self.S / (4.0 * self.df)) * torch.complex(noise[0], noise[1])
        self.rng = rng

    def thetas(self, n):
        near = _near(self.params, self.theta0, self.rng, n // 2)
        return np.ascontiguousarray(np.concatenate([_draws(self.params, self.rng, n - n // 2), near]))

    def strain(self, th):
        """h_i(f) of one parameter vector, [detector, frequency]."""
        C, tau, P = _template(torch.from_numpy(np.asarray(th)[None]).cuda(), self.f, self)
        ph = P[0][None] + self.f[None] * tau[0][:, None]
        return C[0][:, None] * (self.f ** (-7.0 / 6.0)) * _cis(ph)


def _context(ev, **sampler):
    ctx = swig.Context(torch.cuda.current_device())
    ctx.set_grid(ev.f_min, ev.f_max, ev.df)
    data = ev.data.cpu().numpy()
    for i, site in enumerate(ev.sites):
        ctx.set_detector(i, *site)
        ctx.set_data(i, data[i])
        ctx.set_psd(i, ev.psds[i])
    ctx.set_time_ref(ev.gmst)
    ctx.set_prior(ev.params)
    ctx.set_sampler(**sampler)
    return ctx


def prepare(case, seed):
    kind = case["kind"]
    if kind == "retrain":
        rng = np.random.default_rng([seed, 23])
        n, d = case["n"], case["d"]
        t = rng.random(n)  # live points along a curved, correlated ridge of the unit cube
        u = 0.5 + 0.05 * rng.standard_normal((n, d)) + 0.1 * np.outer(t, np.arange(d) % 3 - 1)
        u[:, 0] = 0.2 + 0.6 * t
        u[:, 1] = 0.5 + 0.25 * np.sin(3.0 * t) + 0.02 * rng.standard_normal(n)
        ctx = swig.Context(torch.cuda.current_device())
        return {"case": case, "ctx": ctx, "u": np.clip(u, 0.0, 1.0), "params": ctx.mlp_init(int(seed))}
    ev = _Event(case, seed)
    if kind == "run":
        het = dict(likelihood=swig.LIKE_HET, het_bins=case["bins"], het_fiducial=ev.theta0) if case["bins"] else {}
        return {"case": case, "ctx": _context(ev, nlive=case["nlive"], nrep=case["nlive"] // 10, seed=int(seed),
                                              max_iter=case["iters"], **het)}
    opts = dict(nlive=1000, nrep=100)
    if kind == "fp64":
        opts["precision"] = swig.PREC_FP64
    if kind == "het":
        opts.update(likelihood=swig.LIKE_HET, het_bins=case["bins"], het_spacing=case["spacing"],
                    het_fiducial=ev.theta0, tmarg_nodes=case.get("nodes", 0))
    th = ev.thetas(case["n"])
    state = {"case": case, "ctx": _context(ev, **opts), "theta": th}
    if case["api"] != "host":
        state["theta"] = torch.from_numpy(th).cuda()
        state["out"] = torch.empty(case["n"], dtype=torch.float64, device="cuda")
    if case["api"] == "noalloc":  # prepared ahead, as this entry point asks
        state["ctx"].loglike_batch(th[:1])
    return state


def run(state):
    case, ctx = state["case"], state["ctx"]
    if case["kind"] == "retrain":
        params, rows = ctx.mlp_train(state["u"], state["params"], case["steps"], lr=1e-3)
        return {"params": params, "rows": rows}
    if case["kind"] == "run":
        r = ctx.run()
        theta, logl, logw = ctx.get_samples()
        return {"theta": theta, "logl": logl, "logw": logw, "logz": r.logz, "n_evals": r.n_evals,
                "n_sweep_evals": r.n_sweep_evals}
    if case["api"] == "host":
        return ctx.loglike_batch(state["theta"])
    call = ctx.loglike_batch_noalloc if case["api"] == "noalloc" else ctx.loglike_batch_dev
    call(state["theta"].data_ptr(), case["n"], state["out"].data_ptr(), torch.cuda.current_stream().cuda_stream)
    return state["out"]


def work(case):
    """Per bin one phase (about 14 operations), per bin and detector a time
    shift, a sine, a cosine and a complex multiply-add (12); the weighted data
    are read once.  Heterodyned: per bin edge and detector the same and the
    contraction (30), summary data of 28 bytes per bin and detector; with t_c
    marginalised the eight-point spreading and the FFT on top."""
    kind = case["kind"]
    if kind == "retrain":
        n, layers = case["n"], 13 * 256 + 256 * 256 + 256 * 26
        return {"bytes": 8.0 * n * case["d"] + 4.0 * n * 26 + 2 * 4.0 * 76058,
                "flops": 6.0 * case["steps"] * n * layers + 2.0 * n * layers + 3.0 * n * n * case["d"]}
    bins, dets = int(case["seconds"] * (case["f_max"] - 20.0)) + 1, case["dets"]
    if kind == "run":
        # start, then about 280 full evaluations of each of the nrep chains per iteration
        evals = case["nlive"] * (1 + 28 * case["iters"])
        if case["bins"]:
            return {"bytes": 28.0 * case["bins"] * dets, "flops": evals * case["bins"] * (14.0 + 42.0 * dets)}
        return {"bytes": 8.0 * bins * dets, "flops": evals * bins * (14.0 + 12.0 * dets)}
    n = case["n"]
    io = 8.0 * 14 * n
    if kind == "het":
        b = case["bins"]
        flops = n * b * (14.0 + 42.0 * dets)
        if case["marg"] == "time":
            flops += n * (32.0 * b + 20.0 * case["nodes"] * math.log2(2 * case["nodes"]))
        return {"bytes": io + 28.0 * b * dets, "flops": flops}
    size = 16.0 if kind == "fp64" else 8.0
    return {"bytes": io + size * bins * dets, "flops": n * bins * (14.0 + 12.0 * dets)}


# ---------------------------------------------------------------------------
# The likelihoods in FP64
# ---------------------------------------------------------------------------
MTSUN, C_SI, MPC = 4.925490947641266978e-6, 299792458.0, 3.0856775814913673e22
EULER = 0.57721566490153286061


def _cis(cycles):
    """exp(-2 pi i cycles)."""
    a = 2.0 * math.pi * (cycles - torch.round(cycles))
    return torch.complex(torch.cos(a), -torch.sin(a))


def _template(th, f, ev):
    """TaylorF2 with aligned spins and tides, (2,2) mode: h_i(f) = C_i f^(-7/6)
    exp(-2 pi i (P(f) + f tau_i)).  th: [n, 13]; returns C [n, detector], tau
    [n, detector], P [n, frequency] in cycles."""
    mc, q, c1, c2, l1, l2, dl, inc, psi, ra, dec, tc, phic = (th[:, j] for j in range(13))
    m1, m2 = 1.0 / (1.0 + q), q / (1.0 + q)
    eta, d = m1 * m2, m1 - m2
    pim = math.pi * MTSUN * mc * eta ** (-0.6)
    so = (113.0 / 12.0 * m1**2 + 6.25 * eta) * c1 + (113.0 / 12.0 * m2**2 + 6.25 * eta) * c2
    a2 = 3715.0 / 756.0 + 55.0 / 9.0 * eta
    a3 = -16.0 * math.pi + 4.0 * so
    a4 = 15293365.0 / 508032.0 + 27145.0 / 504.0 * eta + 3085.0 / 72.0 * eta**2 - 98.75 * eta * c1 * c2
    a5 = math.pi * (38645.0 / 756.0 - 65.0 / 9.0 * eta)
    a6 = (11583231236531.0 / 4694215680.0 - 640.0 / 3.0 * math.pi**2 - 6848.0 / 21.0 * EULER
          + (-15737765635.0 / 3048192.0 + 2255.0 / 12.0 * math.pi**2) * eta + 76055.0 / 1728.0 * eta**2
          - 127825.0 / 1296.0 * eta**3)
    a7 = math.pi * (77096675.0 / 254016.0 + 378515.0 / 1512.0 * eta - 74045.0 / 756.0 * eta**2)
    ls, ld = l1 + l2, l1 - l2
    lt = 8.0 / 13.0 * ((1.0 + 7.0 * eta - 31.0 * eta**2) * ls + d * (1.0 + 9.0 * eta - 11.0 * eta**2) * ld)
    dlt = 0.5 * (d * (1.0 - 13272.0 / 1319.0 * eta + 8944.0 / 1319.0 * eta**2) * ls
                 + (1.0 - 15910.0 / 1319.0 * eta + 32850.0 / 1319.0 * eta**2 + 3380.0 / 1319.0 * eta**3) * ld)
    a10, a12 = -19.5 * lt, -3115.0 / 64.0 * lt + 6595.0 / 364.0 * d * dlt
    v = (pim[:, None] * f[None]) ** (1.0 / 3.0)
    lv = torch.log(v)
    e = lambda a: a[:, None]  # noqa: E731
    psum = (1.0 + v**2 * (e(a2) + v * (e(a3) + v * (e(a4) + v * (
        e(a5) * (1.0 + 3.0 * (lv + 0.5 * math.log(6.0))) + v * (
            e(a6) - 6848.0 / 21.0 * (math.log(4.0) + lv) + v * (e(a7) + v**3 * (e(a10) + v**2 * e(a12)))))))))
    P = 3.0 / (256.0 * math.pi) / e(eta) / v**5 * psum - 0.125
    amp = math.sqrt(5.0 / 24.0) * math.pi ** (-2.0 / 3.0) * (MTSUN * mc) ** (5.0 / 6.0) * C_SI / MPC / dl
    lon = ra - ev.gmst
    sl, cl, sd, cd, sp, cp = lon.sin(), lon.cos(), dec.sin(), dec.cos(), psi.sin(), psi.cos()
    east, north = torch.stack([-sl, cl, 0 * sl], 1), torch.stack([-sd * cl, -sd * sl, cd], 1)
    X = -cp[:, None] * east + sp[:, None] * north
    Y = sp[:, None] * east + cp[:, None] * north
    n = torch.stack([cd * cl, cd * sl, sd], 1)
    ci = inc.cos()
    C, tau = [], []
    for vertex, x, y in ev.sites:
        D = torch.from_numpy(0.5 * (np.outer(x, x) - np.outer(y, y))).cuda()
        fp = (X @ D * X).sum(1) - (Y @ D * Y).sum(1)
        fx = 2.0 * (X @ D * Y).sum(1)
        proj = torch.complex(0.5 * (1.0 + ci**2) * fp, -ci * fx)
        C.append(amp * proj * torch.complex(phic.cos(), phic.sin()))
        tau.append(tc - (n @ torch.from_numpy(np.asarray(vertex)).cuda()) / C_SI)
    return torch.stack(C, 1), torch.stack(tau, 1), P


def _marginal(ev, z, hh, dd):
    """log L from Z = <d|h> (complex), <h|h> and <d|d>; d_L marginalised: Z and
    <h|h> are those of the template at 1 Mpc."""
    marg = ev.case["marg"]
    if ev.params[12].mode != si.MODE_MARG:
        core = lambda x, s: s * x  # noqa: E731
        x = z.real
    else:
        core = lambda x, s: s * x + torch.log(torch.special.i0e(s * x))  # noqa: E731
        x = z.abs()
    if marg != "distance":
        return core(x, torch.ones_like(x)) - 0.5 * hh - 0.5 * dd
    p = ev.params[6]
    peak, sig = torch.clamp(x, min=0.0) / hh, 14.0 / torch.sqrt(hh)
    lo, hi = 1.0 / p.hi, 1.0 / p.lo
    a, b = torch.clamp(peak - sig, min=lo), torch.clamp(peak + sig, max=hi)
    a, b = torch.where(peak > hi, torch.clamp(hi - sig, min=lo), a), torch.where(peak < lo, torch.clamp(lo + sig, max=hi), b)
    g, w = np.polynomial.legendre.leggauss(400)
    g, w = torch.from_numpy(g).cuda(), torch.from_numpy(w).cuda()
    u = 0.5 * (a + b)[:, None] + 0.5 * (b - a)[:, None] * g[None]
    dens = math.log(3.0 / (p.hi**3 - p.lo**3)) - 4.0 * torch.log(u)  # p(d) ~ d^2, d = 1 / u
    expo = core(x[:, None], u) - 0.5 * hh[:, None] * u**2 + dens
    return torch.logsumexp(expo + torch.log(w)[None], 1) + torch.log(0.5 * (b - a)) - 0.5 * dd


def _exact_full(ev, th):
    w = 4.0 * ev.df / ev.S
    dd = (w * ev.data.abs() ** 2).sum()
    D = w * ev.data.conj() * ev.f ** (-7.0 / 6.0)
    K = (w * ev.f ** (-7.0 / 3.0)).sum(1)
    out, step = [], max(1, int(2.5e7 // ev.f.numel()))
    for a in range(0, len(th), step):
        C, tau, P = _template(th[a:a + step], ev.f, ev)
        z = 0.0
        for i in range(len(ev.sites)):
            z = z + C[:, i] * (D[i] * _cis(P + ev.f * tau[:, i:i + 1])).sum(1)
        out.append(_marginal(ev, z, (C.abs() ** 2 * K).sum(1), dd))
    return torch.cat(out)


def _edges(f, bins, spacing):
    """Grid indices of the heterodyne's bin edges: equal steps of the largest
    dephasing, or geometric, each at the first grid frequency at or above."""
    if spacing:
        idx = np.searchsorted(f, 10.0 ** (math.log10(f[0]) + np.arange(bins + 1) * (math.log10(f[-1] / f[0]) / bins)))
    else:
        g = sum((-1.0 if p < 0 else 1.0) * (f / (f[0] if p < 0 else f[-1])) ** p
                for p in (-5.0 / 3.0, -2.0 / 3.0, 1.0, 5.0 / 3.0, 7.0 / 3.0))
        idx = np.searchsorted(g, g[0] + np.arange(bins + 1) * ((g[-1] - g[0]) / bins))
    idx[0], idx[-1] = 0, len(f) - 1
    return np.unique(np.minimum(idx, len(f) - 1))


def _exact_het(ev, th):
    case, th, fid = ev.case, th.clone(), ev.theta0.copy()
    if ev.params[12].mode == si.MODE_MARG:
        th[:, 12] = fid[12] = 0.0
    if case["marg"] == "time":
        th[:, 11] = fid[11]
    idx = _edges(ev.freqs, case["bins"], case["spacing"])
    nb = len(idx) - 1
    which = torch.from_numpy(np.minimum(np.searchsorted(idx, np.arange(len(ev.freqs)), side="right") - 1, nb - 1)).cuda()
    fe = ev.f[torch.from_numpy(idx).cuda()]
    off = ev.f - (0.5 * (fe[1:] + fe[:-1]))[which]
    w = 4.0 * ev.df / ev.S
    h0 = ev.strain(fid)
    total = lambda v: torch.zeros(nb, dtype=v.dtype, device="cuda").index_add_(0, which, v)  # noqa: E731
    fidt = torch.from_numpy(fid[None]).cuda()
    C0, tau0, P0 = _template(fidt, fe, ev)
    C, tau, P = _template(th, fe, ev)
    width = fe[1:] - fe[:-1]
    z, hh, y = 0.0, 0.0, 0.0
    for i in range(len(ev.sites)):
        dh, h2 = ev.data[i].conj() * h0[i] * w[i], h0[i].abs() ** 2 * w[i]
        A0, A1, B0, B1 = total(dh), total(dh * off), total(h2), total(h2 * off)
        r = (C[:, i] / C0[0, i])[:, None] * _cis(P - P0 + fe * (tau[:, i] - tau0[0, i])[:, None])
        r0, r1 = 0.5 * (r[:, :-1] + r[:, 1:]), (r[:, 1:] - r[:, :-1]) / width
        z = z + (A0 * r0 + A1 * r1).sum(1)
        hh = hh + (B0 * r0.abs() ** 2 + 2.0 * B1 * (r0 * r1.conj()).real).sum(1)
        g = torch.zeros(nb + 1, dtype=A0.dtype, device="cuda")
        g[:-1] += 0.5 * A0 - A1 / width
        g[1:] += 0.5 * A0 + A1 / width
        y = y + g * r
    dd = (w * ev.data.abs() ** 2).sum()
    if case["marg"] != "time":
        return _marginal(ev, z, hh, dd)
    n, p = case["nodes"], ev.params[11]
    t = p.lo + (torch.arange(n, dtype=torch.float64, device="cuda") + 0.5) * ((p.hi - p.lo) / n) - fid[11]
    zt = y @ _cis(fe[:, None] * t[None])
    x = zt.abs()
    return torch.logsumexp(x + torch.log(torch.special.i0e(x)), 1) - math.log(n) - 0.5 * hh - 0.5 * dd


def exact(case, seed):
    if case["kind"] in ("run", "retrain"):
        return None
    ev = _Event(case, seed)
    th = torch.from_numpy(ev.thetas(case["n"])).cuda()
    if case["marg"] == "distance":
        th[:, 6] = 1.0
    if ev.params[12].mode == si.MODE_MARG:
        th[:, 12] = 0.0
    out = _exact_het(ev, th) if case["kind"] == "het" else _exact_full(ev, th)
    return out.cpu().numpy() if case["api"] == "host" else out
