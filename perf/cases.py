"""The work a user has this library do, as cases that can be timed: log-likelihoods of one field in both
precisions, gradients, kriging, Fisher information and batches of replicate fields, from the smallest to
the largest sizes the library is used at.

A case is a dict of plain values.  ``prepare`` makes its inputs on the GPU from a seed, ``run`` makes one
pass through the public entry points, ``exact`` evaluates the same quantities in plain 64-bit torch.

Inputs: locations on the jittered grid of ``synth.jittered_grid`` (+-0.4 of a cell, x index fastest), cut
after n points; data z from a spectral simulation of the Matern field (random frequencies of its spectral
density), so that z has the smoothness and range of the field it is evaluated under; theta moved a little
around the case's by the seed, as the steps of a fit do.
"""
from __future__ import annotations

import math
import weakref

import numpy as np
import torch

import paper_1908_06936_gb300 as exa
from paper_1908_06936_gb300 import autograd

RADIUS = 6371.0       # km, the library's default sphere for the great-circle metric
FEATURES = 1024       # frequencies of the spectral simulation


def listed():
    return [
        # One evaluation on a small field, as every step of a fit to one of the smallest replicates: latency.
        {"name": "loglik_fp64_n400", "kind": "loglik", "prec": "fp64", "n": 400, "beta": 0.1, "nu": 0.5},
        # One evaluation of the paper's single-field example size, in the default precision.
        {"name": "loglik_fp64_n1600", "kind": "loglik", "prec": "fp64", "n": 1600, "beta": 0.1, "nu": 0.5},
        # A field on the sphere with measurement noise (great-circle distances, a nugget), as for station data.
        {"name": "loglik_sphere_n3721", "kind": "loglik", "prec": "fp64", "n": 3721, "beta": 300.0, "nu": 0.5,
         "metric": 1, "nugget": 0.05},
        # One evaluation on a large field in the default precision; the size is no multiple of any tile.
        {"name": "loglik_fp64_n12300", "kind": "loglik", "prec": "fp64", "n": 12300, "beta": 0.03, "nu": 1.0},
        # One step of a fit to a field of 40,000 points (the derivative-free MLE workload), mixed precision.
        {"name": "loglik_mixed_n40000", "kind": "loglik", "prec": "tf32x3", "n": 40000, "beta": 0.1, "nu": 0.5},
        # The largest field one GPU is used for, mixed precision.
        {"name": "loglik_mixed_n90000", "kind": "loglik", "prec": "tf32x3", "n": 90000, "beta": 0.03, "nu": 1.0},
        # One step of a gradient-based fit through torch.autograd (l forward, dl/dtheta backward), FP64.
        {"name": "grad_fp64_n6400", "kind": "grad", "prec": "fp64", "n": 6400, "beta": 0.1, "nu": 0.5},
        # The same step in mixed precision on a larger field.
        {"name": "grad_mixed_n10000", "kind": "grad", "prec": "tf32x3", "n": 10000, "beta": 0.1, "nu": 0.5},
        # A map: kriging means and variances at 2,048 new points from 10,000 observations.
        {"name": "predict_n10000_m2048", "kind": "predict", "prec": "fp64", "n": 10000, "m": 2048, "beta": 0.1,
         "nu": 0.5},
        # Standard errors of the fitted parameters after a fit: the Fisher information.
        {"name": "fisher_n1600", "kind": "fisher", "prec": "fp64", "n": 1600, "beta": 0.1, "nu": 0.5},
        # A step of a replicate study, exact: fields of 400 to 6,400 points evaluated in one call.
        {"name": "batched_fp64_32", "kind": "batched", "prec": "fp64", "reps": 32, "lo": 20, "hi": 80, "shape": 1,
         "beta": 0.1, "nu": 0.5},
        # The full replicate study of 256 fields, mixed precision on the tensor cores.
        {"name": "batched_mixed_256", "kind": "batched", "prec": "tf32x3", "reps": 256, "lo": 20, "hi": 80,
         "shape": 1, "beta": 0.1, "nu": 0.5},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the ranges above; no drawn case costs more than the largest listed one of its kind."""
    kind = rng.choice(["loglik", "loglik", "sphere", "mixed", "mixed", "grad", "grad_mixed", "predict", "fisher",
                       "batched", "batched_mixed"])
    nu = rng.choice([0.5, 0.5, 0.8, 1.0])
    # the range in units of the field's side, the smoother the shorter (as fits of rough and smooth fields give)
    beta = round(rng.uniform(0.03, 0.15) if nu < 0.75 else rng.uniform(0.02, 0.05), 4)
    case = {"prec": "fp64", "beta": beta, "nu": nu}
    if kind == "loglik":
        case.update(kind="loglik", n=_log_int(rng, 100, 12300))
    elif kind == "sphere":
        case.update(kind="loglik", n=_log_int(rng, 400, 6400), beta=round(rng.uniform(100.0, 500.0), 1),
                    metric=1, nugget=round(rng.uniform(0.01, 0.1), 3))
    elif kind == "mixed":
        case.update(kind="loglik", prec="tf32x3", n=_log_int(rng, 1600, 40000))
    elif kind == "grad":
        case.update(kind="grad", n=_log_int(rng, 400, 6400))
    elif kind == "grad_mixed":
        case.update(kind="grad", prec="tf32x3", n=_log_int(rng, 1600, 10000))
    elif kind == "predict":
        case.update(kind="predict", n=_log_int(rng, 400, 10000), m=_log_int(rng, 50, 2048))
    elif kind == "fisher":
        case.update(kind="fisher", n=_log_int(rng, 100, 1600))
    else:
        case.update(kind="batched", reps=rng.randint(4, 32) if kind == "batched" else rng.randint(16, 256),
                    prec="fp64" if kind == "batched" else rng.choice(["tf32x3", "tf32x3", "fp32"]), lo=20,
                    hi=rng.randint(40, 80), shape=rng.randint(1, 1000))
        if case["prec"] == "fp32":
            case["reps"] = min(case["reps"], 64)
    return case


# --- inputs ------------------------------------------------------------------------------------------

def _theta(case, rng):
    """(sigma^2, beta, nu) of one step of a fit around the case's parameters."""
    u = rng.uniform(-1.0, 1.0, 3)
    return (math.exp(0.1 * u[0]), case["beta"] * math.exp(0.1 * u[1]), case["nu"] * math.exp(0.04 * u[2]))


def _locations(n, gen, sphere):
    m = math.isqrt(n - 1) + 1
    u = (torch.rand(m * m, 2, dtype=torch.float64, device="cuda", generator=gen) - 0.5) * 0.8
    k = torch.arange(m * m, device="cuda")
    s = ((torch.stack([k % m, k // m], 1) + 0.5 + u) / m)[:n]
    if sphere:  # longitudes and latitudes of a region about 2,000 km wide
        s = torch.stack([s[:, 0] * 24.0 - 12.0, s[:, 1] * 20.0 + 30.0], 1)
    return s.contiguous()


def _field(locs, theta, rng, sphere, nugget=0.0):
    """A realisation of the Matern field at locs: FEATURES cosines with frequencies of its spectral density
    (a bivariate t of 2 nu degrees of freedom, scale 1 / beta)."""
    s = locs
    if sphere:  # the tangent plane of the region, in km
        rad = math.pi / 180.0
        s = torch.stack([locs[:, 0] * (rad * RADIUS * math.cos(40.0 * rad)), locs[:, 1] * (rad * RADIUS)], 1)
    w = rng.standard_normal((FEATURES, 2)) / (theta[1] * np.sqrt(rng.chisquare(2.0 * theta[2], (FEATURES, 1))))
    w = torch.as_tensor(w, device="cuda")
    phase = torch.as_tensor(rng.uniform(0.0, 2.0 * math.pi, FEATURES), device="cuda")
    z = torch.empty(len(s), dtype=torch.float64, device="cuda")
    for i in range(0, len(s), 16384):
        z[i:i + 16384] = torch.cos(s[i:i + 16384, :1] * w[:, 0] + s[i:i + 16384, 1:] * w[:, 1] + phase).sum(1)
    z *= math.sqrt(2.0 * theta[0] / FEATURES)
    # what the finite set of frequencies leaves out: variation below the grid's resolution
    z += 0.05 * torch.as_tensor(rng.standard_normal(len(s)), device="cuda")
    if nugget:
        z += math.sqrt(nugget) * torch.as_tensor(rng.standard_normal(len(s)), device="cuda")
    return z.contiguous()


def _inputs(case, seed):
    rng = np.random.default_rng(seed)
    gen = torch.Generator(device="cuda").manual_seed(seed)
    sphere = case.get("metric", 0) == 1
    if case["kind"] == "batched":
        sides = np.random.default_rng(case["shape"]).integers(case["lo"], case["hi"] + 1, size=case["reps"])
        ns = [int(m) * int(m) for m in sides]
        thetas = [_theta(case, rng) for _ in ns]
        locs = [_locations(n, gen, False) for n in ns]
        return {"ns": ns, "locs": locs, "z": [_field(s, t, rng, False) for s, t in zip(locs, thetas)],
                "theta": torch.tensor(thetas, dtype=torch.float64, device="cuda")}
    theta = _theta(case, rng)
    locs = _locations(case["n"], gen, sphere)
    out = {"locs": locs, "z": _field(locs, theta, rng, sphere, case.get("nugget", 0.0)), "theta": theta}
    if case["kind"] == "predict":
        out["new"] = torch.rand(case["m"], 2, dtype=torch.float64, device="cuda", generator=gen)
    return out


# A program keeps one context and evaluates many fields with it: the states of one case share theirs while
# any of them is in use (its workspace at n = 90,000 is half of the GPU's memory).
_contexts = weakref.WeakValueDictionary()


def _context(case):
    key = repr(sorted(case.items()))
    ctx = _contexts.get(key)
    if ctx is None:
        ctx = _contexts[key] = exa.Context()
        if case.get("metric") or case.get("nugget"):
            ctx.check(exa.exa_ctx_set_model(ctx.handle, case.get("nugget", 0.0), case.get("metric", 0), RADIUS))
    return ctx


def prepare(case, seed):
    state = dict(_inputs(case, seed), case=case, ctx=_context(case), prec=exa.PREC[case["prec"]])
    if case["kind"] == "grad":
        state["param"] = torch.tensor(state["theta"], dtype=torch.float64, requires_grad=True)
    elif case["kind"] == "batched":
        state["loglik"] = torch.empty(case["reps"], dtype=torch.float64, device="cuda")
        state["status"] = torch.empty(case["reps"], dtype=torch.int32, device="cuda")
    return state


def run(state):
    kind, ctx = state["case"]["kind"], state["ctx"]
    if kind == "loglik":
        r = ctx.loglik_ex(state["locs"], state["z"], state["theta"], state["prec"])
        return np.array([r["loglik"], r["logdet"], r["quad"]])
    if kind == "grad":
        state["param"].grad = None
        l = autograd.loglik(state["param"], state["locs"], state["z"], ctx, state["prec"])
        l.backward()
        return {"loglik": l.detach(), "grad": state["param"].grad}
    if kind == "predict":
        mean, var = ctx.predict(state["locs"], state["z"], state["theta"], state["new"])
        return {"mean": mean, "var": var}
    if kind == "fisher":
        return {"fisher": ctx.fisher(state["locs"], state["theta"])}
    ctx.check(exa.exa_loglik_batched(ctx.handle, len(state["ns"]), state["ns"], state["locs"], state["z"],
                                     state["theta"], state["prec"], state["loglik"], state["status"]))
    return {"loglik": state["loglik"], "status": state["status"]}


def work(case):
    """Floating-point operations of the contractions and the bytes of inputs and outputs: a matrix of
    covariances need never leave the chip, so it is in neither."""
    kind = case["kind"]
    if kind == "batched":
        sides = np.random.default_rng(case["shape"]).integers(case["lo"], case["hi"] + 1, size=case["reps"])
        n = sides.astype(np.float64) ** 2
        return {"bytes": float(24.0 * n.sum() + 36.0 * len(n)), "flops": float((n ** 3).sum() / 3.0)}
    n = float(case["n"])
    b = 24.0 * n + 24.0
    if kind == "loglik":
        return {"bytes": b, "flops": n ** 3 / 3.0}
    if kind == "grad":  # the factor and Sigma^-1
        return {"bytes": b + 32.0, "flops": n ** 3}
    if kind == "fisher":  # the factor, Sigma^-1 and three symmetric products with it
        return {"bytes": 16.0 * n + 72.0, "flops": 7.0 * n ** 3}
    return {"bytes": b + 32.0 * case["m"], "flops": n ** 3 / 3.0 + n * n * case["m"]}


# --- the same quantities in plain 64-bit torch ---------------------------------------------------------

def _distance(a, b, case):
    if case.get("metric", 0) == 1:
        rad = math.pi / 180.0
        lon, lat = (a[:, None, 0] - b[None, :, 0]) * rad, (a[:, None, 1] - b[None, :, 1]) * rad
        h = torch.sin(0.5 * lat) ** 2 + torch.cos(a[:, None, 1] * rad) * torch.cos(b[None, :, 1] * rad) * torch.sin(
            0.5 * lon) ** 2
        return 2.0 * RADIUS * torch.asin(torch.sqrt(h.clamp(max=1.0)))
    return torch.sqrt((a[:, None, 0] - b[None, :, 0]) ** 2 + (a[:, None, 1] - b[None, :, 1]) ** 2)


def _bessel(nus, x, derivative=False):
    """e^x K_nu(x) for each nu, and e^x dK_nu/dnu of the first: the trapezoid rule on
    int_0^inf exp(-x (cosh t - 1)) cosh(nu t) dt, whose error is far below rounding for this step."""
    h = 1.0 / 16.0
    low = max(float(x.min()), 1e-8)
    steps = int(math.acosh(1.0 + 800.0 / low) / h) + 1
    out = [torch.full_like(x, 0.5) for _ in nus]
    der = torch.zeros_like(x)
    for k in range(1, steps + 1):
        t = k * h
        e = torch.exp(x * (-2.0 * math.sinh(0.5 * t) ** 2))
        for o, nu in zip(out, nus):
            o.add_(e, alpha=math.cosh(nu * t))
        if derivative:
            der.add_(e, alpha=t * math.sinh(nus[0] * t))
    return [o * h for o in out], der * h


def _covariance(a, b, theta, case, derivatives=False):
    """Eq. 3 between two sets of points, with its derivatives in (sigma^2, beta, nu) if asked for."""
    s2, beta, nu = theta
    c = 2.0 ** (1.0 - nu) / math.gamma(nu)
    out = torch.empty(len(a), len(b), dtype=torch.float64, device="cuda")
    der = [torch.empty_like(out) for _ in range(2)] if derivatives else []
    for i in range(0, len(a), 1024):
        x = _distance(a[i:i + 1024], b, case) / beta
        zero = x == 0.0
        x = torch.where(zero, torch.ones_like(x), x)
        if nu == 0.5 and not derivatives:
            v = torch.exp(-x)
        else:
            (k, *km), kd = _bessel([nu, nu - 1.0][:1 + derivatives], x, derivatives)
            pre = c * x ** nu * torch.exp(-x)
            v = pre * k
            if derivatives:
                digamma = float(torch.special.digamma(torch.tensor(nu, dtype=torch.float64)))
                der[0][i:i + 1024] = torch.where(zero, 0.0, s2 * pre * km[0] * x / beta)
                der[1][i:i + 1024] = torch.where(
                    zero, 0.0, s2 * (v * (torch.log(x) - math.log(2.0) - digamma) + pre * kd))
        out[i:i + 1024] = s2 * torch.where(zero, 1.0, v)
    return (out, [out / s2] + der) if derivatives else out


def _evaluate(locs, z, theta, case):
    """l, log|Sigma| and z^T Sigma^-1 z, with the Cholesky factor."""
    sigma = _covariance(locs, locs, theta, case)
    sigma.diagonal().add_(case.get("nugget", 0.0))
    factor = torch.linalg.cholesky(sigma)
    y = torch.linalg.solve_triangular(factor, z[:, None], upper=False)
    logdet, quad = 2.0 * float(factor.diagonal().log().sum()), float((y * y).sum())
    return -0.5 * (len(locs) * math.log(2.0 * math.pi) + logdet + quad), logdet, quad, factor


def exact(case, seed):
    if case["kind"] != "batched" and case["n"] > 16000:
        return None  # a 64-bit factorisation of this size takes longer than is given
    d = _inputs(case, seed)
    if case["kind"] == "batched":
        ls = [_evaluate(s, z, tuple(t), case)[0] for s, z, t in zip(d["locs"], d["z"], d["theta"].tolist())]
        return {"loglik": np.array(ls), "status": None}
    locs, z, theta = d["locs"], d["z"], d["theta"]
    if case["kind"] == "fisher":
        sigma, ders = _covariance(locs, locs, theta, case, True)
        factor = torch.linalg.cholesky(sigma)
        m = [torch.cholesky_solve(x, factor) for x in ders]
        return {"fisher": np.array([[0.5 * float((p * q.T).sum()) for q in m] for p in m])}
    l, logdet, quad, factor = _evaluate(locs, z, theta, case)
    if case["kind"] == "loglik":
        return np.array([l, logdet, quad])
    a = torch.cholesky_solve(z[:, None], factor)
    if case["kind"] == "grad":
        inverse = torch.cholesky_inverse(factor)
        _, ders = _covariance(locs, locs, theta, case, True)
        return {"loglik": np.array(l), "grad": np.array([0.5 * float(((a @ a.T - inverse) * x).sum()) for x in ders])}
    cross = _covariance(locs, d["new"], theta, case)
    y = torch.linalg.solve_triangular(factor, cross, upper=False)
    return {"mean": (cross.T @ a)[:, 0], "var": theta[0] - (y * y).sum(0)}
