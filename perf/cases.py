"""Performance cases: the calls that a user of the library makes, over the sizes they are made at.

Each case is one pass through the public Python face (paper_2003_12861_gb300.api):
likelihood passes (small, large, all-FP32, any-graph, user-defined densities,
batches of toys), fits, toy generation with its histograms, the binned
likelihood and the learned-start network's training step.  Events are drawn
here, from the densities themselves (an inverse-CDF table); exact() restates
every likelihood in 64-bit torch.
"""
import math

import numpy as np
import torch

from paper_2003_12861_gb300 import api
from paper_2003_12861_gb300 import workloads as W

DEV = "cuda"

# Generating values, in theta order (the benchmark workloads' own).
TRUE = {
    "gauss_poly1": [5.0, 0.5, 0.3, -0.05],
    "decay": [1.5, 0.0, 0.05, -0.2, 0.05, 0.2],
    "decay_generic": [1.5, 0.0, 0.05, -0.2, 0.05, 0.8],
    "prod3": [5.28, 0.015, 0.4, -0.3, 1.5, 0.0, 0.05, -0.2, 0.05, 0.2, 0.1, 0.3],
    "expr_mix": [5.28, 0.012, 0.45, -0.2, 1.5, 1.2],
}
# How far theta is moved from them where the likelihood is evaluated (a
# minimiser's trial points near the end of a fit).
STEP = {
    "gauss_poly1": [0.02, 0.02, 0.01, 0.003],
    "decay": [0.03, 0.002, 0.002, 0.02, 0.02, 0.01],
    "decay_generic": [0.03, 0.002, 0.002, 0.02, 0.02, 0.01],
    "prod3": [0.0005, 0.0005, 0.01, 0.02, 0.03, 0.002, 0.002, 0.02, 0.02, 0.01, 0.02, 0.02],
    "expr_mix": [0.0005, 0.0005, 0.01, 0.02, 0.05, 0.05],
}
SPEC = {
    "gauss_poly1": W.gauss_poly1_model,
    "decay": W.decay_model,
    "decay_generic": W.decay_generic_model,
    "prod3": W.prod3_model,
    "expr_mix": W.expr_mix_model,
}
# Floating-point operations per event of the density and its gradient (an
# exponential, logarithm, power or reciprocal counted as 10).
FLOPS = {"gauss_poly1": 60, "decay": 70, "decay_generic": 70, "prod3": 190, "expr_mix": 170}
OBS = {"gauss_poly1": 1, "decay": 1, "decay_generic": 1, "prod3": 3, "expr_mix": 2}


def listed():
    return [
        # the smallest likelihood call: a minimiser's step on a small dataset, where latency is everything
        {"name": "gauss_poly1_1e4", "do": "nll_grad", "model": "gauss_poly1", "n": 10000, "f32": False},
        # an ordinary unbinned fit's step
        {"name": "decay_1e7", "do": "nll_grad", "model": "decay", "n": 10000000, "f32": False},
        # the headline workload: three FP32 observables, 12 parameters, the largest dataset
        {"name": "prod3_1e8_f32", "do": "nll_grad", "model": "prod3", "n": 100000000, "f32": True},
        # a graph without a program of its own: the FP64 interpreter
        {"name": "decay_generic_4e6", "do": "nll_grad", "model": "decay_generic", "n": 4000003, "f32": False},
        # user-defined densities (postfix programs) with numerical normalisation
        {"name": "expr_mix_1e6", "do": "nll_grad", "model": "expr_mix", "n": 1000001, "f32": False},
        # likelihood values of a batch of ragged toys (a profile scan's or a test statistic's step; no gradient)
        {"name": "toys_nll_512", "do": "toys_nll", "model": "decay", "sets": 512},
        # one dataset's fit with its covariance
        {"name": "fit_decay_1e6", "do": "fit", "model": "decay", "n": 1000003},
        # a batched toy study
        {"name": "fit_toys_256", "do": "fit_toys", "model": "decay", "sets": 256},
        # toy Monte Carlo: generation and the histograms that the learned start reads
        {"name": "gen_toys_1024", "do": "gen", "model": "decay", "sets": 1024, "f32": False},
        # binned likelihood of the observed data alone (host arrays, as a minimiser calls it)
        {"name": "binned_1", "do": "binned", "channels": 28, "bins": 50, "sets": 1, "host": True},
        # and of a batch of toy datasets on the device
        {"name": "binned_1024", "do": "binned", "channels": 28, "bins": 50, "sets": 1024, "host": False},
        # one optimiser step of the learned-start network (the trainer's default batch)
        {"name": "mlp_step_1024", "do": "mlp", "rows": 1024, "hidden": 128, "layers": 3},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    do = rng.choice(["nll_grad", "nll_grad", "nll_grad", "toys_nll", "fit", "fit_toys", "gen", "binned", "mlp"])
    if do == "nll_grad":
        model = rng.choice(["gauss_poly1", "decay", "prod3", "decay_generic", "expr_mix"])
        most = {"gauss_poly1": 2e7, "decay": 2e7, "prod3": 5e7, "decay_generic": 4e6, "expr_mix": 2e6}[model]
        return {"do": do, "model": model, "n": _log_int(rng, 1e3, most), "f32": rng.random() < 0.5}
    if do == "toys_nll":
        return {"do": do, "model": rng.choice(["decay", "gauss_poly1"]), "sets": _log_int(rng, 2, 1024)}
    if do == "fit":
        return {"do": do, "model": "decay", "n": _log_int(rng, 3e5, 3e6)}
    if do == "fit_toys":
        return {"do": do, "model": rng.choice(["decay", "gauss_poly1"]), "sets": _log_int(rng, 2, 512)}
    if do == "gen":
        return {"do": do, "model": rng.choice(["decay", "gauss_poly1", "prod3"]), "sets": _log_int(rng, 1, 1500),
                "f32": rng.random() < 0.3}
    if do == "binned":
        return {"do": do, "channels": rng.randint(1, 28), "bins": rng.randint(5, 50), "sets": _log_int(rng, 1, 2048),
                "host": rng.random() < 0.3}
    return {"do": do, "rows": _log_int(rng, 33, 4096), "hidden": rng.choice([64, 96, 128, 256]),
            "layers": rng.randint(1, 4)}


# ------------------------------------------------- densities in 64-bit torch

def _phi(x):
    return 0.5 * torch.special.erfc(-x * math.sqrt(0.5))


def _norm_mass(a, b):
    """Phi(b) - Phi(a), from the smaller tails."""
    up = _phi(-a) - _phi(-b)
    return torch.where(a > 0, up, _phi(b) - _phi(a))


def _gauss(x, mu, sg, lo, hi, at):
    mass = _norm_mass((lo - mu) / sg, (hi - mu) / sg)
    u = (x - at(mu)) / at(sg)
    return torch.exp(-0.5 * u * u) / at(sg * math.sqrt(2 * math.pi) * mass)


def _gaussexp_shape(t, tau, mu, sg):
    u, s = (t - mu) / sg, sg / tau
    z = (s - u) * math.sqrt(0.5)
    zp, zn = torch.clamp(z, min=0.0), torch.clamp(z, max=0.0)
    above = 0.5 * torch.exp(-0.5 * u * u) * torch.special.erfcx(zp)
    below = 0.5 * torch.exp(torch.where(z > 0, torch.zeros_like(z), s * (0.5 * s - u))) * torch.special.erfc(zn)
    return torch.where(z > 0, above, below)


def _gaussexp(t, tau, mu, sg, lo, hi, at):
    mass = _norm_mass((lo - mu) / sg, (hi - mu) / sg)
    end = [_gaussexp_shape(torch.full_like(tau, v), tau, mu, sg) for v in (lo, hi)]
    norm = tau * (mass - end[1] + end[0])
    return _gaussexp_shape(t, at(tau), at(mu), at(sg)) / at(norm)


def _cheb(x, cs, lo, hi, at):
    y = (2 * x - lo - hi) / (hi - lo)
    terms, ints = [y, 2 * y * y - 1], [0.0, -2.0 / 3.0]
    shape, norm = 1.0, 2.0
    for c, t, i in zip(cs, terms, ints):
        shape = shape + at(c) * t
        norm = norm + c * i
    return shape / at(0.5 * (hi - lo) * norm)


def _poly(x, cs, lo, hi, at):
    shape, norm = 1.0, hi - lo
    for k, c in enumerate(cs, 1):
        shape = shape + at(c) * x ** k
        norm = norm + c * (hi ** (k + 1) - lo ** (k + 1)) / (k + 1)
    return shape / at(norm)


def _decay(t, p, at, sig=None):
    f = p[5] if sig is None else sig
    return at(f) * _gaussexp(t, p[0], p[1], p[2], 0.0, 10.0, at) + at(1 - f) * _cheb(t, p[3:5], 0.0, 10.0, at)


def _factors(model, x, p, at):
    """The model's density, as its factors (one per observable)."""
    if model == "gauss_poly1":
        return [at(p[2]) * _gauss(x[0], p[0], p[1], 0.0, 10.0, at) + at(1 - p[2]) * _poly(x[0], p[3:], 0.0, 10.0, at)]
    if model == "decay":
        return [_decay(x[0], p, at)]
    if model == "decay_generic":
        return [_decay(x[0], p, at, 1 - p[5])]
    if model == "prod3":
        mass = at(p[2]) * _gauss(x[0], p[0], p[1], 5.2, 5.4, at) + at(1 - p[2]) * _cheb(x[0], p[3:4], 5.2, 5.4, at)
        return [mass, _decay(x[1], p[4:10], at), _poly(x[2], p[10:], -1.0, 1.0, at)]
    # expr_mix: a Cauchy line on a straight line, times t^a exp(-b t)
    m0, gam, f = p[0], p[1], p[2]
    line_norm = (torch.atan((5.4 - m0) / gam) - torch.atan((5.2 - m0) / gam)) / gam
    line = 1.0 / ((x[0] - at(m0)) ** 2 + at(gam) ** 2) / at(line_norm)
    mass = at(f) * line + at(1 - f) * _cheb(x[0], p[3:4], 5.2, 5.4, at)
    node, weight = np.polynomial.legendre.leggauss(160)
    tt = torch.as_tensor(2.6 + 2.4 * node, dtype=torch.float64, device=p[4].device)
    ww = torch.as_tensor(2.4 * weight, dtype=torch.float64, device=p[4].device)
    norm = (ww * torch.exp(p[4][..., None] * torch.log(tt) - p[5][..., None] * tt)).sum(-1)
    return [mass, torch.exp(at(p[4]) * torch.log(x[1]) - at(p[5]) * x[1]) / at(norm)]


RANGE = {
    "gauss_poly1": [(0.0, 10.0)],
    "decay": [(0.0, 10.0)],
    "decay_generic": [(0.0, 10.0)],
    "prod3": [(5.2, 5.4), (0.0, 10.0), (-1.0, 1.0)],
    "expr_mix": [(5.2, 5.4), (0.2, 5.0)],
}


# --------------------------------------------------------------- the inputs

def _columns(model, n, seed, f32):
    """n events per observable from the model's density at its generating
    values (inverse CDF on 2^16 cells), on the GPU."""
    gen = torch.Generator(DEV).manual_seed(seed)
    p = [torch.tensor(v, dtype=torch.float64) for v in TRUE[model]]
    grids = [torch.linspace(lo, hi, 200001, dtype=torch.float64) for lo, hi in RANGE[model]]
    dens = _factors(model, grids, p, lambda v: v)
    cols = []
    for c, (g, d) in enumerate(zip(grids, dens)):
        x, y = g.numpy(), d.numpy()
        cdf = np.concatenate([[0.0], np.cumsum(0.5 * (y[1:] + y[:-1]))])
        tab = torch.as_tensor(np.interp(np.linspace(0.0, 1.0, 65537), cdf / cdf[-1], x), device=DEV)
        out = torch.empty(n, dtype=torch.float32 if f32 else torch.float64, device=DEV)
        lo, hi = RANGE[model][c]
        if f32:  # the nearest float of an end may lie outside the range
            lo, hi = float(np.nextafter(np.float32(lo), np.float32(np.inf))), float(np.nextafter(np.float32(hi), np.float32(-np.inf)))
        for a in range(0, n, 1 << 24):
            b = min(n, a + (1 << 24))
            u = torch.rand(b - a, dtype=torch.float64, device=DEV, generator=gen) * 65536
            i = u.long().clamp_(max=65535)
            out[a:b] = torch.clamp(torch.lerp(tab[i], tab[i + 1], u - i), lo, hi)
        cols.append(out)
    return cols


def _theta(model, seed, sets=None):
    rng = np.random.Generator(np.random.PCG64(seed + 31))
    shape = (len(TRUE[model]),) if sets is None else (sets, len(TRUE[model]))
    return np.asarray(TRUE[model]) + np.asarray(STEP[model]) * rng.uniform(-1.0, 1.0, shape)


def _mean_sizes(sets, seed):
    """Toy sizes, log-uniform between 1e3 and 1e5 events."""
    rng = np.random.Generator(np.random.PCG64(seed + 17))
    return np.exp(rng.uniform(math.log(1e3), math.log(1e5), sets))


def _offsets(sets, seed):
    return np.concatenate([[0], np.cumsum(np.rint(_mean_sizes(sets, seed)).astype(np.int64))])


def _binned_spec(case, seed):
    """A HistFactory-like model (per channel 8 samples, each with 10 normsys and
    20 histosys modifiers out of 253 shared nuisances, 3 free scales), counts
    drawn around its expectation, and one parameter point per dataset."""
    rng = np.random.Generator(np.random.PCG64(seed + 5))
    C, B, S, samples, nuis, n_hs, n_ns = case["channels"], case["bins"], case["sets"], 8, 253, 20, 10
    x = (np.arange(B) + 0.5) / B
    N = C * samples
    amp = 10 ** rng.uniform(0.5, 3.0, N)
    h = amp[:, None] * np.exp(-x * rng.uniform(0.5, 4.0, N)[:, None]) * (1 + 0.2 * np.sin(6.28 * x * rng.uniform(0.5, 2, N)[:, None]))
    sig = np.arange(N) % samples == 0
    bump = amp[:, None] * (np.exp(-0.5 * ((x - rng.uniform(0.3, 0.7, N)[:, None]) / rng.uniform(0.05, 0.15, N)[:, None]) ** 2) + 1e-3)
    h[sig] = bump[sig]
    order = np.argsort(rng.random((N, nuis)), axis=1)
    ns_par, hs_par = 3 + order[:, :n_ns], 3 + order[:, n_ns:n_ns + n_hs]
    k_lo, k_hi = rng.uniform(0.85, 0.99, (N, n_ns)), rng.uniform(1.01, 1.15, (N, n_ns))
    tilt = rng.uniform(-0.05, 0.05, (N, n_hs, 1)) * (x - 0.5) + rng.uniform(-0.02, 0.02, (N, n_hs, 1))
    lo = h[:, None] * (1 - tilt - rng.uniform(0, 0.01, (N, n_hs, 1)))
    hi = h[:, None] * (1 + tilt + rng.uniform(0, 0.01, (N, n_hs, 1)))
    mods = []
    for s in range(N):
        if s % samples < 3:
            mods.append((s, 0, s % samples, 1.0, 1.0, None, None))
        mods += [(s, 1, int(ns_par[s, j]), float(k_lo[s, j]), float(k_hi[s, j]), None, None) for j in range(n_ns)]
        mods += [(s, 2, int(hs_par[s, j]), 1.0, 1.0, lo[s, j], hi[s, j]) for j in range(n_hs)]
    spec = {"n_bins": C * B, "bin0": [(s // samples) * B for s in range(N)], "nominal": list(h),
            "constrained": [False] * 3 + [True] * nuis, "modifiers": mods}
    theta = rng.normal(0.0, 0.5, (S, 3 + nuis))
    theta[:, :3] = rng.uniform(0.8, 1.2, (S, 3))
    counts = rng.poisson(np.tile(h.reshape(C, samples, B).sum(1).reshape(-1), (S, 1))).astype(np.float64)
    parts = {"h": h, "ns_par": ns_par, "k_lo": k_lo, "k_hi": k_hi, "hs_par": hs_par, "lo": lo, "hi": hi}
    return spec, counts, theta, parts


def _mlp_dims(case):
    return [64] + [case["hidden"]] * case["layers"] + [6]


def _mlp_inputs(case, seed):
    """Histogram-like rows, standardised targets, and weights at the trainer's scale."""
    g = torch.Generator(DEV).manual_seed(seed)
    centre = torch.rand(case["rows"], 1, device=DEV, generator=g) * 64
    x = torch.exp(-torch.arange(64, device=DEV) / (4 + centre)) + 0.05 * torch.rand(case["rows"], 64, device=DEV, generator=g)
    x = (x / x.sum(1, keepdim=True)).contiguous()
    t = torch.randn(case["rows"], 6, device=DEV, generator=g)
    rng = np.random.Generator(np.random.PCG64(seed + 3))
    dims = _mlp_dims(case)
    parts = []
    for a, b in zip(dims, dims[1:]):
        parts += [rng.uniform(-1.0, 1.0, a * b) / math.sqrt(a), rng.uniform(-0.1, 0.1, b)]
    return x, t, np.concatenate(parts).astype(np.float32)


# ------------------------------------------------------------- the interface

def prepare(case, seed):
    do = case["do"]
    if do in ("nll_grad", "fit"):
        model = api.Model.from_spec(SPEC[case["model"]]())
        data = api.Data.from_torch(model, _columns(case["model"], case["n"], seed, case.get("f32", False)))
        return {"do": do, "model": model, "data": data, "theta": _theta(case["model"], seed)}
    if do in ("toys_nll", "fit_toys"):
        model = api.Model.from_spec(SPEC[case["model"]]())
        off = _offsets(case["sets"], seed)
        data = api.Data.from_torch(model, _columns(case["model"], int(off[-1]), seed, False), off)
        return {"do": do, "model": model, "data": data, "theta": _theta(case["model"], seed, case["sets"])}
    if do == "gen":
        return {"do": do, "model": api.Model.from_spec(SPEC[case["model"]]()), "seed": seed,
                "theta": _theta(case["model"], seed, case["sets"]), "mean": _mean_sizes(case["sets"], seed),
                "f32": [case["f32"]] * OBS[case["model"]], "col": OBS[case["model"]] // 2}
    if do == "binned":
        spec, counts, theta, _ = _binned_spec(case, seed)
        state = {"do": do, "model": api.BinnedModel(spec), "host": case["host"], "counts": counts, "theta": theta}
        if not case["host"]:
            S, P = theta.shape
            state["counts"] = torch.as_tensor(counts, device=DEV)
            state["theta"] = torch.as_tensor(theta, device=DEV)
            state["out"] = torch.zeros(S, 1 + P, dtype=torch.float64, device=DEV)
            state["flags"] = torch.zeros(S, dtype=torch.int32, device=DEV)
        return state
    x, t, w = _mlp_inputs(case, seed)
    net = api.MLP(n_hidden=case["hidden"], n_hidden_layers=case["layers"])
    net.set_params(w)
    return {"do": do, "net": net, "x": x, "t": t, "grad": torch.zeros(net.n_params, device=DEV)}


def run(state):
    do = state["do"]
    if do == "nll_grad":
        return list(api.nll_grad(state["model"], state["data"], state["theta"]))
    if do == "toys_nll":
        return [api.nll(state["model"], state["data"], state["theta"])]
    if do == "fit":
        r = api.fit(state["model"], state["data"])
        return [r["theta"], r["nll"], r["cov"], r["n_evals"], r["status"]]
    if do == "fit_toys":
        r = api.fit(state["model"], state["data"], want_cov=False)
        return [r["theta"], r["nll"], r["n_evals"], r["status"]]
    if do == "gen":
        data = api.generate_toys(state["model"], state["theta"], state["seed"], state["mean"], f32=state["f32"])
        hist = torch.empty(data.n_sets, 64, dtype=torch.float32, device=DEV)
        api.hist64(state["model"], data, state["col"], hist)
        off = data.offsets()
        data.close()
        return [off, hist]
    if do == "binned":
        if state["host"]:
            return list(state["model"].nll_grad(state["counts"], state["theta"]))
        state["model"].nll_grad_async(state["counts"], state["theta"], state["out"], state["flags"])
        return [state["out"], state["flags"]]
    loss = state["net"].grad(state["x"], state["t"], state["grad"])
    state["net"].adam(1e-3)
    return [loss, state["grad"]]


def work(case):
    do = case["do"]
    if do == "nll_grad":
        n, width = case["n"], (4 if case["f32"] else 8) * OBS[case["model"]]
        return {"bytes": n * width, "flops": n * FLOPS[case["model"]]}
    if do == "toys_nll":  # 2.15e4 events a toy on average; the density alone is about half of the work
        n = 21500 * case["sets"]
        return {"bytes": 8 * n, "flops": n * FLOPS[case["model"]] / 2}
    if do == "fit":  # about 30 evaluations to the minimum and 12 for the covariance
        return {"bytes": 8 * case["n"], "flops": 42 * case["n"] * FLOPS[case["model"]]}
    if do == "fit_toys":  # about 40 evaluations a toy
        n = 21500 * case["sets"]
        return {"bytes": 8 * n, "flops": 40 * n * FLOPS[case["model"]]}
    if do == "gen":  # every event written once, one column read again for the histograms; about 3 tries an event
        n, width = 21500 * case["sets"], 4 if case["f32"] else 8
        return {"bytes": n * width * (OBS[case["model"]] + 1), "flops": n * 100 * OBS[case["model"]]}
    if do == "binned":  # two multiply-adds a histosys term and bin, forward and backward
        C, B, S = case["channels"], case["bins"], case["sets"]
        terms = C * 8 * 20 * B
        return {"bytes": 16 * terms + 8 * S * (C * B + 2 * 256), "flops": S * (8 * terms + 40 * C * B)}
    dims = _mlp_dims(case)
    weights = sum(a * b for a, b in zip(dims, dims[1:]))
    return {"bytes": case["rows"] * 70 * 4 + 8 * weights, "flops": 6 * case["rows"] * weights}


# ------------------------------------------------------ the same in 64 bits

def _exact_nll_grad(model, cols, theta):
    p = [torch.tensor(float(v), dtype=torch.float64, device=DEV, requires_grad=True) for v in theta]
    n = cols[0].numel()
    nll, grad = 0.0, np.zeros(len(p))
    for a in range(0, n, 1 << 22):
        x = [c[a:a + (1 << 22)].double() for c in cols]
        f = _factors(model, x, p, lambda v: v)
        s = -sum(torch.log(v).sum() for v in f)
        grad += torch.stack(torch.autograd.grad(s, p)).cpu().numpy()
        nll += float(s.detach())
    return nll, grad


def _exact_fit(model, col, theta):
    """The minimum by Newton's method (64-bit gradient and Hessian) from the
    generating values, the NLL there and the inverse Hessian."""
    theta = np.array(theta, dtype=np.float64)
    n = len(theta)
    for it in range(12):
        g, H, f = np.zeros(n), np.zeros((n, n)), 0.0
        for a in range(0, col.numel(), 1 << 20):
            p = [torch.tensor(float(v), dtype=torch.float64, device=DEV, requires_grad=True) for v in theta]
            s = -torch.log(_factors(model, [col[a:a + (1 << 20)]], p, lambda v: v)[0]).sum()
            first = torch.autograd.grad(s, p, create_graph=True)
            for i in range(n):
                H[i] += torch.stack(torch.autograd.grad(first[i], p, retain_graph=True)).detach().cpu().numpy()
            g += torch.stack(first).detach().cpu().numpy()
            f += float(s.detach())
        step = np.linalg.solve(H, g)
        if g @ step < 1e-16:
            break
        theta = theta - step
    return theta, f, np.linalg.inv(H)


def exact(case, seed):
    do = case["do"]
    if do == "nll_grad":
        cols = _columns(case["model"], case["n"], seed, case["f32"])
        nll, grad = _exact_nll_grad(case["model"], cols, _theta(case["model"], seed))
        return [np.float64(nll), grad]
    if do == "toys_nll":
        off = _offsets(case["sets"], seed)
        cols = _columns(case["model"], int(off[-1]), seed, False)
        th = _theta(case["model"], seed, case["sets"])
        out = np.zeros(case["sets"])
        for a in range(0, case["sets"], 64):  # 64 sets at a time
            b = min(case["sets"], a + 64)
            idx = torch.repeat_interleave(torch.arange(b - a, device=DEV), torch.as_tensor(np.diff(off[a:b + 1]), device=DEV))
            p = [torch.as_tensor(th[a:b, k].copy(), device=DEV) for k in range(th.shape[1])]
            x = [c[int(off[a]):int(off[b])] for c in cols]
            logp = sum(torch.log(f) for f in _factors(case["model"], x, p, lambda v: v[idx]))
            ends = np.cumsum([0] + list(np.diff(off[a:b + 1])))
            out[a:b] = [-float(logp[int(i):int(j)].sum()) for i, j in zip(ends[:-1], ends[1:])]
        return [out]
    if do == "fit":
        col = _columns(case["model"], case["n"], seed, False)[0]
        theta, f, cov = _exact_fit(case["model"], col, TRUE[case["model"]])
        return [theta[None], np.array([f]), cov[None], None, None]
    if do == "binned":
        spec, counts, theta, q = _binned_spec(case, seed)
        C, B, S, P = case["channels"], case["bins"], case["sets"], theta.shape[1]
        up = lambda v: torch.as_tensor(np.ascontiguousarray(v), device=DEV)  # noqa: E731
        h, lo, hi = up(q["h"]), up(q["lo"]), up(q["hi"])
        la, lb = 0.5 * (up(q["k_hi"]).log() - up(q["k_lo"]).log()), 0.5 * (up(q["k_hi"]).log() + up(q["k_lo"]).log())
        ha, hb = 0.5 * (hi - lo), 0.5 * (hi + lo) - h[:, None]
        nll, grad = np.zeros(S), np.zeros((S, P))
        for a in range(0, S, 64):
            th = up(theta[a:a + 64]).requires_grad_(True)
            n = up(counts[a:a + 64])
            g = torch.where(th.abs() <= 1, th * th, 2 * th.abs() - 1)
            eta = torch.exp((la * th[:, up(q["ns_par"])] + lb * g[:, up(q["ns_par"])]).sum(-1))
            scale = torch.cat([th[:, :3], torch.ones(th.shape[0], 5, dtype=torch.float64, device=DEV)], 1).repeat(1, C)
            al, gl = th[:, up(q["hs_par"])], g[:, up(q["hs_par"])]
            shape = h + torch.einsum("snj,njb->snb", al, ha) + torch.einsum("snj,njb->snb", gl, hb)
            nu = ((eta * scale)[..., None] * shape).view(-1, C, 8, B).sum(2).reshape(-1, C * B)
            f = (nu - n * torch.log(nu)).sum(1) + 0.5 * (th[:, 3:] ** 2).sum(1)
            grad[a:a + 64] = torch.autograd.grad(f.sum(), th)[0].cpu().numpy()
            nll[a:a + 64] = f.detach().cpu().numpy()
        return [nll, grad] if case["host"] else [np.concatenate([nll[:, None], grad], 1), None]
    if do == "mlp":
        x, t, w = _mlp_inputs(case, seed)
        w = torch.as_tensor(w.astype(np.float64), device=DEV).requires_grad_(True)
        dims, at, y = _mlp_dims(case), 0, x.double()
        for k, (a, b) in enumerate(zip(dims, dims[1:])):
            y = y @ w[at:at + a * b].view(a, b) + w[at + a * b:at + a * b + b]
            at += a * b + b
            if k < len(dims) - 2:
                y = torch.nn.functional.gelu(y)
        loss = ((y - t.double()) ** 2).mean()
        return [float(loss.detach()), torch.autograd.grad(loss, w)[0]]
    # a toy fit may end in one of several minima, and generated toys are what
    # the generator's bits make them: no 64-bit value of their own
    return None
