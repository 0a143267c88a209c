"""The work a user has this library do, as cases to measure.

Each case is one call (or, for the server, one batch of calls) through the public Python
binding, on inputs shaped like a quantitative-MRI study: protocols, prior bounds, proposal
steps and noise levels are those of ``paper_2511_22094_gb300.workloads``, sizes run from the
paper's smallest speed test (100 voxels, Sec. 2.5) to a masked whole volume.

The measured data are simulated here, in plain float64 torch, so that inputs do not depend on
the library.
"""
import math
import random

import numpy as np
import torch

from paper_2511_22094_gb300 import gac
from paper_2511_22094_gb300 import workloads as W

_BASE = {"monoexp": W.MONOEXP_4K, "mwi3": W.MWI3_1M, "smt": W.SMT_1P5M, "axcal": W.AXCAL_250K}

#: FP32 operations of one likelihood per measured value (model and residual) and per evaluation
#: (set-up, proposal, random numbers, decision), evaluated the cheapest way known for each model.
_OPS = {"monoexp": (4, 120), "mwi3": (15, 500), "smt": (34, 170), "axcal": (45, 190)}


# ----------------------------------------------------------------- the cases
def _mh(model, n, chains, iterations, **kw):
    c = {"path": "mh", "model": model, "n": n, "chains": chains, "iterations": iterations,
         "burnin": iterations // 10, "thin": 100, "echoes": len(_BASE[model].acq), "all_moments": False,
         "adapt": 0, "host": False, "fp32": False}
    c.update(kw)
    return c


def listed():
    return [
        # myelin-water mapping of a masked whole volume (the paper's method, Table 1's thinning)
        {"name": "mwi3_volume", **_mh("mwi3", 200_000, 4, 2500)},
        # one slice's brain mask, with burn-in step adaptation, moments over every state and R-hat
        {"name": "mwi3_slice", **_mh("mwi3", 12_345, 4, 2000, all_moments=True, adapt=50)},
        # a region of interest, called as the README does: host arrays in, host arrays out
        {"name": "mwi3_roi", **_mh("mwi3", 301, 4, 5000, host=True)},
        # R2* mapping of one 64 x 64 slice: the repository's 4,096-voxel workload
        {"name": "monoexp_4k", **_mh("monoexp", 4096, 1, 2000, burnin=500, thin=5)},
        # diffusion (Standard Model) whole volume at 2 mm
        {"name": "smt_volume", **_mh("smt", 150_000, 4, 2500)},
        # the paper's smallest speed test: 100 samples, Table 1's 4 chains x 25,000 iterations
        {"name": "axcal_100", **_mh("axcal", 100, 4, 25_000)},
        # axon-diameter mapping of a white-matter mask
        {"name": "axcal_mask", **_mh("axcal", 25_001, 4, 5000)},
        # the ensemble sampler, Table 1's 50 walkers
        {"name": "ensemble_mwi3", "path": "ensemble", "model": "mwi3", "n": 3001, "chains": 50,
         "iterations": 1000, "burnin": 100, "thin": 100, "echoes": 24},
        # gradient fit of a whole volume: L1 loss, 3D total variation on the myelin-water amplitude
        {"name": "fit_mwi3_volume", "path": "fit", "model": "mwi3", "nx": 96, "ny": 96, "nz": 60,
         "echoes": 24, "iterations": 100, "l1": True, "tv": 1e-3, "mask": True},
        # gradient fit of a cropped region, least squares, many updates
        {"name": "fit_monoexp_crop", "path": "fit", "model": "monoexp", "nx": 37, "ny": 41, "nz": 9,
         "echoes": 12, "iterations": 300, "l1": False, "tv": 0.0, "mask": False},
        # a study's queue: ten jobs of mixed models and sizes handed to the server at once
        {"name": "serve_queue", "path": "serve", "jobs": 10, "n": 30_000, "iterations": 1500, "mix": 1},
        # simulated signals for a Monte Carlo study (the sampler's own arithmetic)
        {"name": "simulate_mwi3", "path": "forward", "model": "mwi3", "n": 500_000, "echoes": 24},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    path = rng.choice(["mh", "mh", "mh", "mh", "ensemble", "fit", "serve", "forward"])
    model = rng.choice(["monoexp", "mwi3", "smt", "axcal"])
    echoes = {"monoexp": rng.randint(6, 24), "mwi3": rng.randint(12, 32), "smt": 6, "axcal": 48}[model]
    cost = {"monoexp": 1, "mwi3": 3, "smt": 1.5, "axcal": 3.5}[model]  # relative time per likelihood
    if path == "mh":
        chains = rng.choice([1, 2, 3, 4, 4, 4])
        iterations = _log_int(rng, 500, 10_000)
        n = _log_int(rng, 100, min(250_000, 5e9 / cost / chains / iterations))
        return _mh(model, n, chains, iterations, echoes=echoes, thin=rng.choice([5, 10, 25, 100]) if n < 20_000 else 100,
                   all_moments=rng.random() < 0.25, adapt=rng.choice([0, 0, 50]), host=n < 20_000 and rng.random() < 0.3,
                   fp32=rng.random() < 0.1)
    if path == "ensemble":
        walkers = rng.choice([20, 32, 50, 64])
        iterations = _log_int(rng, 200, 2000)
        n = _log_int(rng, 100, max(200, min(20_000, 1e9 / cost / walkers / iterations)))
        return {"path": "ensemble", "model": model, "n": n, "chains": walkers, "iterations": iterations,
                "burnin": iterations // 10, "thin": rng.choice([20, 50, 100]), "echoes": echoes}
    if path == "fit":
        model = rng.choice(["monoexp", "mwi3", "smt"])
        echoes = {"monoexp": rng.randint(6, 24), "mwi3": rng.randint(12, 32), "smt": 6}[model]
        s = _log_int(rng, 2000, 600_000)
        nx = rng.randint(12, 110)
        ny = max(4, min(110, int(math.sqrt(s / nx) * rng.uniform(1.0, 2.5))))
        return {"path": "fit", "model": model, "nx": nx, "ny": ny, "nz": max(2, s // (nx * ny)), "echoes": echoes,
                "iterations": rng.choice([50, 100, 150]), "l1": rng.random() < 0.6, "tv": rng.choice([0.0, 1e-3, 1e-2]),
                "mask": rng.random() < 0.5}
    if path == "serve":
        return {"path": "serve", "jobs": rng.randint(2, 12), "n": _log_int(rng, 1000, 25_000),
                "iterations": _log_int(rng, 500, 1500), "mix": rng.randint(2, 10**6)}
    return {"path": "forward", "model": model, "n": _log_int(rng, 1000, 1_000_000), "echoes": echoes}


# -------------------------------------------- protocols and simulated signals
def _acq(model, echoes):
    """`echoes` evenly spaced echo times over the protocol's range; b-values and AxCaliberSMT's
    (b, Delta, delta) triplets as they are."""
    base = _BASE[model].acq
    if model in ("smt", "axcal") or echoes == len(base):
        return list(base)
    return [base[0] + k * (base[-1] - base[0]) / (echoes - 1) for k in range(echoes)]


def _n_meas(model, echoes):
    return {"mwi3": 2 * echoes, "axcal": len(_BASE["axcal"].acq) // 3}.get(model, echoes)


def _g(x):
    """int_0^1 exp(-x u^2) du by 48-point Gauss-Legendre quadrature."""
    u, w = np.polynomial.legendre.leggauss(48)
    out = torch.zeros_like(x)
    for ui, wi in zip((u + 1) / 2, w / 2):
        out += wi * torch.exp(-x * ui**2)
    return out


def _j1p_zeros(count):
    """The first zeros of J1' (Newton on J1'(x) = J0 - J1 / x from McMahon's estimate)."""
    x = (torch.arange(1, count + 1, dtype=torch.float64) - 0.25) * math.pi
    x[0] = 1.8412
    for _ in range(40):
        j0, j1 = torch.special.bessel_j0(x), torch.special.bessel_j1(x)
        d1 = j0 - j1 / x
        x = x - d1 / (-j1 - d1 / x + j1 / x**2)
    return x


def _forward64(model, acq, th):
    """Noise-free measurements [n][M] in float64 (complex echoes as re, im pairs)."""
    if model == "monoexp":
        t = torch.tensor(acq, dtype=torch.float64, device=th.device)
        return th[:, :1] * torch.exp(-th[:, 1:2] * t * 1e-3)
    if model == "mwi3":
        t = torch.tensor(acq, dtype=torch.float64, device=th.device)
        re = im = 0.0
        for j in range(3):
            mag = th[:, j : j + 1] * torch.exp(-t / th[:, 3 + j : 4 + j])
            ang = th[:, 8:9] - (2 * math.pi * 1e-3 * th[:, 6 + j : 7 + j] * t if j < 2 else 0.0)
            re = re + mag * torch.cos(ang)
            im = im + mag * torch.sin(ang)
        return torch.stack([re, im], dim=2).reshape(th.shape[0], -1)
    if model == "smt":
        f, da, dpar, dperp = th[:, :1], th[:, 1:2], th[:, 2:3], th[:, 3:4]
        b = torch.tensor(acq, dtype=torch.float64, device=th.device)
        return f * _g(b * da) + (1 - f) * torch.exp(-b * dperp) * _g(b * (dpar - dperp))
    # AxCaliberSMT: Gaussian-phase cylinders, axial diffusivities 1.7, free water 3 um^2/ms
    x = _j1p_zeros(60).to(th.device)
    r2 = (0.5 * th[:, 0]) ** 2
    fn, fc, der = th[:, 1], th[:, 2], th[:, 3]
    cols, phi = [], {}
    for b, big, small in zip(acq[0::3], acq[1::3], acq[2::3]):
        if (big, small) not in phi:
            s = torch.zeros_like(r2)
            for xm in x.tolist():
                q = xm * xm * 1.7 / r2
                a = q * small
                e = torch.where(a < 1e-2, a * a * (0.5 - a / 6 + a * a / 24), torch.expm1(-a) + a)
                n = 2 * e - torch.exp(-q * (big - small)) * torch.expm1(-a) ** 2
                s += 2 / (1.7**2 * xm**6 * (xm**2 - 1)) * n
            phi[(big, small)] = s * r2**3
        kap = b / (small**2 * (big - small / 3)) * phi[(big, small)]
        cols.append((1 - fc) * (fn * torch.exp(-kap) * _g(b * 1.7 - kap) + (1 - fn) * torch.exp(-b * der) * _g(b * (1.7 - der)))
                    + fc * math.exp(-3.0 * b))
    return torch.stack(cols, dim=1)


def _truths(model, n, gen, dev):
    """True parameters [n][P] from the workloads' ranges."""
    w = _BASE[model]
    lb = torch.tensor(w.lb, dtype=torch.float64, device=dev)
    ub = torch.tensor(w.ub, dtype=torch.float64, device=dev)
    u = torch.rand((n, len(w.lb)), generator=gen, dtype=torch.float64, device=dev)
    if model == "axcal":
        lb = torch.tensor((1.0, 0.3, 0.0, 0.3), dtype=torch.float64, device=dev)
        ub = torch.tensor((10.0, 0.8, 0.2, 1.2), dtype=torch.float64, device=dev)
    th = lb + (ub - lb) * u
    if model == "mwi3":  # myelin-water fraction ~ U(0, 0.3)
        mwf = 0.3 * u[:, 0]
        th[:, 0] = mwf * (th[:, 1] + th[:, 2]) / (1 - mwf)
    return th


def _sigma(model, th):
    """Noise SD per voxel at the workload's SNR."""
    snr = _BASE[model].snr
    if model == "monoexp":
        return (th[:, 0] / snr).float()
    if model == "mwi3":
        return (th[:, :3].sum(1) / snr).float()
    return torch.full((th.shape[0],), 1.0 / snr, dtype=torch.float32, device=th.device)


def _measured(model, acq, n, gen, dev):
    """Truths, noise SD and noisy data [n][M] (float32), simulated in pieces of 65,536 voxels."""
    th = _truths(model, n, gen, dev)
    sig = _sigma(model, th)
    y = torch.cat([_forward64(model, acq, th[i : i + 65536]) for i in range(0, n, 65536)])
    y += sig.double()[:, None] * torch.randn(y.shape, generator=gen, dtype=torch.float64, device=dev)
    return th, sig, y.float().contiguous()


def _register(model, acq):
    w = _BASE[model]
    return gac.gac_model_register(w.kind, acq, w.lb, w.ub, w.step)


# ------------------------------------------------------------------- prepare
def _sampler_outputs(case, dev):
    P, N, C = len(_BASE[case["model"]].lb), case["n"], case["chains"]
    S = gac.n_samples(case["iterations"], case["burnin"], case["thin"])
    out = dict(mean=torch.empty((P, N), dtype=torch.float64, device=dev),
               std=torch.empty((P, N), dtype=torch.float64, device=dev),
               samples=torch.empty((S, C, P, N), dtype=torch.float32, device=dev),
               accept_rate=torch.empty((C, N), dtype=torch.float32, device=dev),
               nonfinite=torch.empty((C, N), dtype=torch.int32, device=dev))
    if case.get("adapt"):
        out["rhat"] = torch.empty((P, N), dtype=torch.float64, device=dev)
        out["step_scale"] = torch.empty((C, N), dtype=torch.float32, device=dev)
    if case.get("all_moments"):  # moments over every state: the samples are not kept
        del out["samples"]
    return out


def _prepare_mh(case, seed, gen, dev):
    acq = _acq(case["model"], case["echoes"])
    _, sig, y = _measured(case["model"], acq, case["n"], gen, dev)
    st = {"mid": _register(case["model"], acq)}
    kw = dict(precision=gac.PREC_FP32 if case["fp32"] else gac.PREC_MIXED,
              moments_mode=gac.MOMENTS_ALL_POSTBURNIN if case["all_moments"] else gac.MOMENTS_THINNED,
              adapt_window=case["adapt"], adapt_target=0.3 if case["adapt"] else 0.0)
    sampler = dict(iterations=case["iterations"], burnin=case["burnin"], thin=case["thin"],
                   n_chains=case["chains"], seed=seed)
    if case["host"]:
        st.update(y=y.cpu().numpy(), sig=sig.cpu().numpy(), kw={**sampler, **kw, "want_samples": not case["all_moments"]})
    else:
        st.update(y=y, sig=sig, out=_sampler_outputs(case, dev), opts=gac.make_opts(**sampler, **kw))
    return st


def _prepare_ensemble(case, seed, gen, dev):
    acq = _acq(case["model"], case["echoes"])
    th, sig, y = _measured(case["model"], acq, case["n"], gen, dev)
    # walkers start in a ball around a first fit, inside the prior box
    w = _BASE[case["model"]]
    lb = torch.tensor(w.lb, dtype=torch.float64, device=dev)
    ub = torch.tensor(w.ub, dtype=torch.float64, device=dev)
    x0 = th[:, None, :] + 0.02 * (ub - lb) * torch.randn((case["n"], case["chains"], len(w.lb)), generator=gen,
                                                        dtype=torch.float64, device=dev)
    x0 = torch.minimum(torch.maximum(x0, lb + 1e-3 * (ub - lb)), ub - 1e-3 * (ub - lb)).float().contiguous()
    opts = gac.make_opts(case["iterations"], case["burnin"], case["thin"], case["chains"], seed)
    return {"mid": _register(case["model"], acq), "y": y, "sig": sig, "x0": x0, "opts": opts,
            "out": _sampler_outputs(case, dev)}


def _fit_inputs(case, seed, dev):
    gen = torch.Generator(device=dev).manual_seed(seed)
    acq = _acq(case["model"], case["echoes"])
    n = case["nx"] * case["ny"] * case["nz"]
    _, sig, y = _measured(case["model"], acq, n, gen, dev)
    w = _BASE[case["model"]]
    lb = torch.tensor(w.lb, dtype=torch.float64, device=dev)
    ub = torch.tensor(w.ub, dtype=torch.float64, device=dev)
    # start anywhere in the middle of the box; weights from the voxel's SNR; an ellipsoidal mask
    theta0 = lb + (ub - lb) * (0.3 + 0.4 * torch.rand((n, len(w.lb)), generator=gen, dtype=torch.float64, device=dev))
    weight = (0.01 / sig).float()
    mask = None
    if case["mask"]:
        ax = [torch.linspace(-1, 1, m, device=dev) for m in (case["nx"], case["ny"], case["nz"])]
        r = ax[0][None, None, :] ** 2 + ax[1][None, :, None] ** 2 + 0.6 * ax[2][:, None, None] ** 2
        mask = (r.reshape(-1) < 1.1).to(torch.uint8).contiguous()
    return acq, y, weight, mask, theta0, lb, ub


def _prepare_fit(case, seed, gen, dev):
    acq, y, weight, mask, theta0, _, _ = _fit_inputs(case, seed, dev)
    opts = gac.make_fit_opts((case["nx"], case["ny"], case["nz"]), loss=gac.FIT_L1 if case["l1"] else gac.FIT_L2,
                             iterations=case["iterations"], learning_rate=0.01, tv_lambda=case["tv"],
                             tv_params=1 if case["tv"] else 0, tv_dims=3)
    return {"mid": _register(case["model"], acq), "y": y, "weight": weight, "mask": mask, "theta0": theta0,
            "theta": torch.empty_like(theta0), "opts": opts,
            "loss": torch.zeros(case["iterations"], dtype=torch.float64, device=dev)}


class _Server:
    """A server that a program keeps for as long as it runs."""

    def __init__(self):
        self.handle = gac.gac_server_create(32 << 30, 64)

    def __del__(self):
        if getattr(self, "handle", None):
            gac.gac_server_destroy(self.handle)


def _serve_jobs(case):
    """The queue's jobs: model, voxels (up to four times apart), chains and iterations."""
    rng = random.Random(case["mix"])
    return [(rng.choice(("monoexp", "mwi3", "smt")), max(1, int(case["n"] * 2 ** rng.uniform(-1, 1))),
             rng.randint(1, 4), max(1, int(case["iterations"] * rng.uniform(0.5, 1.5)))) for _ in range(case["jobs"])]


def _prepare_serve(case, seed, gen, dev):
    jobs = []
    for k, (model, n, chains, iterations) in enumerate(_serve_jobs(case)):
        acq = list(_BASE[model].acq)
        _, sig, y = _measured(model, acq, n, gen, dev)
        P = len(_BASE[model].lb)
        jobs.append({"mid": _register(model, acq), "n": n, "y": y.cpu().numpy(), "sig": sig.cpu().numpy(),
                     "opts": gac.make_opts(iterations, iterations // 10, 100, chains, 1000 * seed + k),
                     "out": dict(mean=np.empty((P, n)), std=np.empty((P, n)),
                                 accept_rate=np.empty((chains, n), np.float32))})
    return {"server": _Server(), "jobs": jobs}


def _prepare_forward(case, seed, gen, dev):
    acq = _acq(case["model"], case["echoes"])
    theta = _truths(case["model"], case["n"], gen, dev).contiguous()
    return {"mid": _register(case["model"], acq), "theta": theta,
            "s": torch.empty((case["n"], _n_meas(case["model"], case["echoes"])), dtype=torch.float64, device=dev)}


_PREPARE = {"mh": _prepare_mh, "ensemble": _prepare_ensemble, "fit": _prepare_fit, "serve": _prepare_serve,
            "forward": _prepare_forward}


def prepare(case, seed):
    dev = torch.device("cuda:0")
    gen = torch.Generator(device=dev).manual_seed(seed)
    return {"path": case["path"], "case": case, **_PREPARE[case["path"]](case, seed, gen, dev)}


# ----------------------------------------------------------------------- run
def run(state):
    case, path = state["case"], state["path"]
    if path == "serve":
        ids = [gac.gac_server_submit(state["server"].handle, j["mid"], j["y"], j["n"], j["sig"], 0.0, j["opts"])
               for j in state["jobs"]]
        for i, j in zip(ids, state["jobs"]):
            gac.gac_server_wait(state["server"].handle, i, 60.0, j["out"])
        return [j["out"] for j in state["jobs"]]
    if path == "mh" and case["host"]:
        return {k: v for k, v in gac.run_host(state["mid"], state["y"], state["sig"], **state["kw"]).items()
                if v is not None}
    stream = torch.cuda.current_stream()
    if path == "mh":
        gac.gac_mcmc_run(state["mid"], state["y"], case["n"], state["sig"], 0.0, None, state["opts"], state["out"], stream)
        return state["out"]
    if path == "ensemble":
        gac.gac_ensemble_run(state["mid"], state["y"], case["n"], state["sig"], 0.0, state["x0"], state["opts"], 2.0,
                             state["out"], stream)
        return state["out"]
    if path == "fit":
        state["theta"].copy_(state["theta0"])
        gac.gac_fit_run(state["mid"], state["y"], state["mask"], state["weight"], state["opts"], state["theta"],
                        state["loss"], stream)
        return {"theta": state["theta"], "loss": state["loss"]}
    gac.gac_forward(state["mid"], state["theta"], case["n"], gac.PREC_MIXED, state["s"], stream)
    return state["s"]


# ---------------------------------------------------------------------- work
def _sampler_work(model, echoes, n, chains, iterations, burnin, thin, samples=True, x0=False):
    P, M = len(_BASE[model].lb), _n_meas(model, echoes)
    per_value, per_eval = _OPS[model]
    stored = gac.n_samples(iterations, burnin, thin) * chains * P * 4 if samples else 0
    return {"bytes": n * (4 * M + 4 + 16 * P + 8 * chains + stored + (4 * chains * P if x0 else 0)),
            "flops": n * chains * iterations * (per_value * M + per_eval)}


def work(case):
    path = case["path"]
    if path == "mh":
        return _sampler_work(case["model"], case["echoes"], case["n"], case["chains"], case["iterations"], case["burnin"],
                             case["thin"], samples=not case["all_moments"])
    if path == "ensemble":
        return _sampler_work(case["model"], case["echoes"], case["n"], case["chains"], case["iterations"], case["burnin"],
                             case["thin"], x0=True)
    if path == "serve":
        jobs = [_sampler_work(m, len(_BASE[m].acq), n, c, it, it // 10, 100, samples=False)
                for m, n, c, it in _serve_jobs(case)]
        return {k: sum(j[k] for j in jobs) for k in ("bytes", "flops")}
    P, M = len(_BASE[case["model"]].lb), _n_meas(case["model"], case["echoes"])
    per_value, per_eval = _OPS[case["model"]]
    if path == "forward":
        return {"bytes": case["n"] * 8 * (P + M), "flops": case["n"] * (per_value * M + per_eval)}
    n = case["nx"] * case["ny"] * case["nz"]
    # parameters in and out once; the model, its Jacobian (about twice the model) and Adam every update
    return {"bytes": n * (4 * M + 16 * P + 5), "flops": n * case["iterations"] * (3 * per_value * M + 12 * P)}


# --------------------------------------------------------------------- exact
def _fit64(case, seed):
    """The fit's Adam iteration in float64 with automatic derivatives."""
    dev = torch.device("cuda:0")
    acq, y, weight, mask, theta0, lb, ub = _fit_inputs(case, seed, dev)
    nx, ny, nz = case["nx"], case["ny"], case["nz"]
    inside = torch.ones(nx * ny * nz, dtype=torch.bool, device=dev) if mask is None else mask.bool()
    idx = inside.nonzero()[:, 0]
    n_mask, M = idx.numel(), y.shape[1]
    grid = inside.reshape(nz, ny, nx)
    pairs = [(grid.narrow(d, 1, grid.shape[d] - 1) & grid.narrow(d, 0, grid.shape[d] - 1)) for d in range(3)]
    yd, wd = y.double(), weight.double()
    u = ((theta0 - lb) / (ub - lb)).clamp(0, 1)
    m1, m2 = torch.zeros_like(u), torch.zeros_like(u)
    hist = []
    for t in range(1, case["iterations"] + 1):
        g, loss = torch.zeros_like(u), 0.0
        for i in idx.split(65536):
            ui = u[i].requires_grad_(True)
            r = wd[i, None] * (yd[i] - _forward64(case["model"], acq, lb + ui * (ub - lb)))
            part = (r.abs().sum() if case["l1"] else (r * r).sum()) / (n_mask * M)
            g[i] = torch.autograd.grad(part, ui)[0]
            loss = loss + part.detach()
        if case["tv"]:
            c = u[:, 0].reshape(nz, ny, nx)
            gc = torch.zeros_like(c)
            for d in range(3):
                k = c.shape[d] - 1
                diff = (c.narrow(d, 1, k) - c.narrow(d, 0, k)) * pairs[d]
                loss = loss + case["tv"] / n_mask * diff.abs().sum()
                gc.narrow(d, 1, k).add_(diff.sign())
                gc.narrow(d, 0, k).sub_(diff.sign())
            g[:, 0] += case["tv"] / n_mask * gc.reshape(-1)
        hist.append(loss)
        m1 = 0.9 * m1 + 0.1 * g
        m2 = 0.999 * m2 + 0.001 * g * g
        step = 0.01 * (m1 / (1 - 0.9**t)) / ((m2 / (1 - 0.999**t)).sqrt() + 1e-8)
        u = torch.where(inside[:, None], (u - step).clamp(0, 1), u)
    theta = torch.where(inside[:, None], lb + u * (ub - lb), theta0)
    return {"theta": theta, "loss": torch.stack([torch.as_tensor(h) for h in hist])}


def exact(case, seed):
    """Signals and fits in float64.  A sampler's outputs have no such value: they are the path of
    a Markov chain whose accept/reject decisions follow from the sampler's own 32-bit
    likelihoods, and a 64-bit chain takes another path of the same distribution."""
    if case["path"] == "forward":
        dev = torch.device("cuda:0")
        gen = torch.Generator(device=dev).manual_seed(seed)
        th = _truths(case["model"], case["n"], gen, dev)
        acq = _acq(case["model"], case["echoes"])
        return torch.cat([_forward64(case["model"], acq, th[i : i + 65536]) for i in range(0, case["n"], 65536)])
    if case["path"] == "fit" and case["nx"] * case["ny"] * case["nz"] * case["iterations"] <= 60_000_000:
        return _fit64(case, seed)
    return None
