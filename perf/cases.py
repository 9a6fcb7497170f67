"""The library's main path as a set of measured cases.

Each case is one call (or the two calls of a likelihood evaluation) through the
public Python binding, as a user's program makes it, over the sizes that the
tests, the benchmark and the parameter sweep of this repository use:

* ``matern``: the covariance matrix of one parameter vector (FP64 plain form,
  FP32 precision form, FP32 with the learned window), n = 500 .. 40,000;
* ``cross``: the m x n cross-covariance between observations and prediction
  points;
* ``batched``: the matrices of a maximum-likelihood sweep in one persistent
  launch;
* ``host``: a matrix delivered to page-locked host memory;
* ``eval``: K_nu(x) of (x, nu) pairs, FP64 or FP32 with either window;
* ``grad``: K, dK/dx and dK/dnu of pairs (gradient-based likelihoods);
* ``loglik``: one likelihood evaluation, the matrix and its Gaussian
  log-likelihood.
"""
from __future__ import annotations

import math
import os

import numpy as np
import torch

import paper_2502_00356_gb300 as bk
from paper_2502_00356_gb300 import inputs

WEIGHTS = os.path.join(os.path.dirname(os.path.abspath(bk.__file__)), "weights", "window_mlp.bkw")


def listed():
    return [
        # the smallest matrices of a sweep: launches and one wave of tiles
        {"name": "matern-f64-777", "kind": "matern", "form": "f64", "n": 777, "beta": 0.1, "nu": 0.8},
        # an ordinary likelihood evaluation's matrix, ragged
        {"name": "matern-f64-4001", "kind": "matern", "form": "f64", "n": 4001, "beta": 0.1, "nu": 2.3},
        # the benchmark's matrix
        {"name": "matern-f64-20000", "kind": "matern", "form": "f64", "n": 20000, "beta": 0.1, "nu": 1.5},
        # the large single-precision matrix
        {"name": "matern-f32-40000", "kind": "matern", "form": "f32", "n": 40000, "beta": 0.05,
         "nu": 2.5},
        # prediction: observations against a set of new points
        {"name": "cross-f64-20000x2003", "kind": "cross", "form": "f64", "m": 20000, "n": 2003,
         "beta": 0.1, "nu": 0.5},
        # a parameter sweep in the fastest form
        {"name": "batched-learned-24", "kind": "batched", "form": "learned", "count": 24},
        # a matrix for a host-side solver
        {"name": "host-f64-6000", "kind": "host", "form": "f64", "n": 6000, "beta": 0.1, "nu": 2.3},
        # bare evaluations: the benchmark's 100,000 pairs
        {"name": "eval-f64-100000", "kind": "eval", "form": "f64", "n": 100000, "nu_hi": 10.0},
        # many pairs in single precision
        {"name": "eval-learned-1e7", "kind": "eval", "form": "learned", "n": 10000000, "nu_hi": 20.0},
        # derivatives for a gradient-based likelihood
        {"name": "grad-f64-100000", "kind": "grad", "form": "f64", "n": 100000, "nu_hi": 10.0},
        # likelihood evaluations: a small data set and an ordinary one
        {"name": "loglik-1000", "kind": "loglik", "form": "f64", "n": 1000, "beta": 0.1, "nu": 0.8},
        {"name": "loglik-8000", "kind": "loglik", "form": "f64", "n": 8000, "beta": 0.1, "nu": 0.5},
    ]


def _log_uniform(rng, lo, hi):
    return int(math.exp(rng.uniform(math.log(lo), math.log(hi + 1))))


def draw(rng):
    kind = rng.choice(("matern", "matern", "cross", "batched", "host", "eval", "eval", "grad",
                       "loglik", "loglik"))
    beta, nu = rng.uniform(0.02, 0.3), rng.uniform(0.3, 3.5)
    if rng.random() < 0.3:
        nu = rng.choice((0.5, 1.5, 2.5))
    if kind == "matern":
        form = rng.choice(("f64", "f64", "f32", "learned"))
        return {"kind": kind, "form": form, "n": _log_uniform(rng, 500, 20000), "beta": beta, "nu": nu}
    if kind == "cross":
        form = rng.choice(("f64", "f64", "f32"))
        return {"kind": kind, "form": form, "m": _log_uniform(rng, 500, 20000),
                "n": _log_uniform(rng, 33, 4000), "beta": beta, "nu": nu}
    if kind == "batched":
        return {"kind": kind, "form": rng.choice(("f64", "f32", "learned")), "count": rng.randint(3, 24)}
    if kind == "host":
        return {"kind": kind, "form": rng.choice(("f64", "f32")), "n": _log_uniform(rng, 500, 6000),
                "beta": beta, "nu": nu}
    if kind == "eval":
        form = rng.choice(("f64", "f32", "learned"))
        return {"kind": kind, "form": form, "n": _log_uniform(rng, 1000, 4000000),
                "nu_hi": rng.choice((10.0, 20.0))}
    if kind == "grad":
        return {"kind": kind, "form": "f64", "n": _log_uniform(rng, 1000, 1000000), "nu_hi": 10.0}
    return {"kind": kind, "form": "f64", "n": _log_uniform(rng, 300, 8000), "beta": rng.uniform(0.05, 0.3),
            "nu": rng.choice((0.5, rng.uniform(0.4, 1.0)))}


# ---------------------------------------------------------------------------
# inputs

def _locs(n, seed, device="cuda"):
    return torch.as_tensor(inputs.morton_sorted(inputs.jittered_grid(n, seed=seed)), device=device)


def _targets(case, seed):
    """Prediction points: uniform in the unit square, in Morton order."""
    return inputs.morton_sorted(np.random.default_rng([seed, 7]).random((2, case["n"])))


def _pairs(case, seed):
    """x log-uniform in [1e-3, 140], nu uniform in [0.05, nu_hi]."""
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    u = torch.rand((2, case["n"]), generator=g, dtype=torch.float64, device="cuda")
    x = torch.exp(math.log(1e-3) + u[0] * math.log(140.0 / 1e-3))
    return x, 0.05 + u[1] * (case["nu_hi"] - 0.05)


def _observations(case, locs, seed):
    """A field with the spectrum of the Matern covariance (a sum of 256 random
    waves) at the locations, and measurement noise."""
    rng = np.random.default_rng([seed, 11])
    k = 256
    w = rng.standard_normal((k, 2)) / (case["beta"] * np.sqrt(rng.chisquare(2 * case["nu"], (k, 1))))
    phase = rng.uniform(0, 2 * math.pi, k)
    t = lambda a: torch.as_tensor(a, device="cuda")
    z = torch.cos(t(w) @ locs + t(phase)[:, None]).sum(0) * math.sqrt(2.0 / k)
    return z + 0.05 * t(rng.standard_normal(case["n"]))


def _instances(case, seed):
    """The sweep's first `count` sizes; parameters and locations from the seed."""
    sizes = [i.n for i in inputs.batched_instances(case["count"])]
    inst = inputs.batched_instances(case["count"], seed=seed, first_instance_seed=seed + 1)
    for i, n in zip(inst, sizes):
        i.n = n
    return inst


def _dtype(form):
    return torch.float64 if form == "f64" else torch.float32


def prepare(case, seed):
    kind, form = case["kind"], case["form"]
    s = {"case": case, "net": bk.LearnedWindow(path=WEIGHTS) if form == "learned" else None}
    s["opts"] = bk.make_opts(learned=s["net"]) if form == "learned" else None
    dt = _dtype(form)
    if kind == "matern":
        s["locs"] = _locs(case["n"], seed)
        s["out"] = torch.empty((case["n"], case["n"]), dtype=dt, device="cuda")
    elif kind == "cross":
        s["locs"] = _locs(case["m"], seed)
        s["targets"] = torch.as_tensor(_targets(case, seed), device="cuda")
        s["out"] = torch.empty((case["n"], case["m"]), dtype=dt, device="cuda")
    elif kind == "batched":
        inst = _instances(case, seed)
        s["items"] = [(torch.as_tensor(i.locations(), device="cuda"), i.sigma2, i.beta, i.nu,
                       torch.empty((i.n, i.n), dtype=dt, device="cuda")) for i in inst]
        s["descs"] = bk.make_descs(s["items"])
        s["plan"] = bk.BatchedPlan([i.n for i in inst], dtype=dt, opts=s["opts"])
    elif kind == "host":
        s["locs"] = _locs(case["n"], seed, "cpu").pin_memory()
        s["out"] = torch.empty((case["n"], case["n"]), dtype=dt, pin_memory=True)
        s["work"] = torch.empty(bk.matern_tile_host_workspace(case["n"], dt, staged=False),
                                dtype=torch.uint8, device="cuda")
    elif kind == "eval":
        s["x"], s["nu"] = _pairs(case, seed)
        s["opts"] = bk.make_opts(compute=bk.BK_F32) if form == "f32" else s["opts"]
        s["out"] = torch.empty(case["n"], dtype=dt, device="cuda")
    elif kind == "grad":
        s["x"], s["nu"] = _pairs(case, seed)
        s["outs"] = [torch.empty(case["n"], dtype=dt, device="cuda") for _ in range(3)]
    else:
        s["locs"] = _locs(case["n"], seed)
        s["z"] = _observations(case, s["locs"], seed)
        s["a"] = torch.empty((case["n"], case["n"]), dtype=dt, device="cuda")
        s["y"] = torch.empty(case["n"], dtype=dt, device="cuda")
        s["out"] = torch.empty(3, dtype=dt, device="cuda")
    return s


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "matern":
        return bk.bk_matern_tile(s["locs"], 1.0, case["beta"], case["nu"], out=s["out"], opts=s["opts"])
    if kind == "cross":
        return bk.bk_matern_tile2(s["locs"], s["targets"], 1.0, case["beta"], case["nu"], out=s["out"],
                                  opts=s["opts"])
    if kind == "batched":
        bk.bk_matern_batched(s["descs"], s["plan"])
        return [it[4] for it in s["items"]]
    if kind == "host":
        return bk.bk_matern_tile_host(s["locs"], 1.0, case["beta"], case["nu"], s["out"], s["work"],
                                      opts=s["opts"])
    if kind == "eval":
        return bk.bk_eval_ex(s["x"], s["nu"], out=s["out"], opts=s["opts"])[0]
    if kind == "grad":
        return bk.bk_eval_grad(s["x"], s["nu"], *s["outs"])
    bk.bk_matern_tile(s["locs"], 1.0, case["beta"], case["nu"], out=s["a"])
    bk.bk_gaussian_loglik(s["a"], s["z"], y=s["y"], out=s["out"])
    return {"out": s["out"], "a": s["a"], "y": s["y"]}


# ---------------------------------------------------------------------------
# What a pass cannot do without: inputs read once, outputs written once, and
# the arithmetic of the results' definition: the squared distance of each
# unordered pair (5) and one smooth function of it (10); for the pairs'
# evaluations an integral of about 15 terms of 4 operations; n^3 / 3 for a
# Cholesky factorisation.

def work(case):
    kind, size = case["kind"], 8 if case["form"] == "f64" else 4
    if kind in ("matern", "host"):
        n = case["n"]
        return {"bytes": size * n * n + 16 * n, "flops": 15 * n * (n + 1) // 2}
    if kind == "cross":
        m, n = case["m"], case["n"]
        return {"bytes": size * m * n + 16 * (m + n), "flops": 15 * m * n}
    if kind == "batched":
        ns = [i.n for i in _instances(case, 0)]
        return {"bytes": sum(size * n * n + 16 * n for n in ns),
                "flops": sum(15 * n * (n + 1) // 2 for n in ns)}
    if kind == "eval":
        return {"bytes": (16 + size) * case["n"], "flops": 60 * case["n"]}
    if kind == "grad":
        return {"bytes": 40 * case["n"], "flops": 120 * case["n"]}
    n = case["n"]  # the matrix written, its lower triangle read and overwritten
    return {"bytes": 16 * n * n + 16 * n, "flops": 15 * n * (n + 1) // 2 + n ** 3 // 3}


# ---------------------------------------------------------------------------
# The same results in plain torch, FP64: the integral by a trapezoid rule on a
# fixed fine grid, the closed forms of half-integer orders.

def _nodes(x_min, h=1.0 / 20):
    """t_j on [0, T], T where e^{-x cosh t} is negligible for every x >= x_min."""
    top = math.acosh(1.0 + 800.0 / x_min) if x_min < 800 else 2.0
    t = torch.arange(0, int(top / h) + 2, dtype=torch.float64, device="cuda") * h
    w = torch.full_like(t, h)
    w[0] = 0.5 * h
    return t, w


def _matern_of(x, nu):
    """2^{1-nu}/Gamma(nu) x^nu K_nu(x), 1 at x = 0."""
    if nu == 0.5:
        return torch.exp(-x)
    if nu == 1.5:
        return (1 + x) * torch.exp(-x)
    if nu == 2.5:
        return (1 + x + x * x / 3) * torch.exp(-x)
    pos = x > 0
    xs = torch.where(pos, x, 1.0)
    t, w = _nodes(float(xs.min()))
    s = torch.zeros_like(xs)
    ch, co = (torch.cosh(t) - 1).tolist(), (torch.cosh(nu * t) * w).tolist()
    for c, f in zip(ch, co):
        s += torch.exp(xs * -c).mul_(f)
    v = s * torch.exp(nu * torch.log(xs) - xs + ((1 - nu) * math.log(2.0) - math.lgamma(nu)))
    return torch.where(pos, v, 1.0)


def _matrix(l1, l2, beta, nu, sigma2, dtype):
    """out[j, i] = M(|l2_j - l1_i|), in slabs of rows."""
    m, n = l1.shape[1], l2.shape[1]
    out = torch.empty((n, m), dtype=dtype, device="cuda")
    rows = max(1, 16000000 // max(m, 1))
    for j in range(0, n, rows):
        d = l2[:, j:j + rows]
        r = torch.sqrt((l1[0][None, :] - d[0][:, None]) ** 2 + (l1[1][None, :] - d[1][:, None]) ** 2)
        out[j:j + rows] = sigma2 * _matern_of(r / beta, nu)
    return out


def _pair_sums(x, nu, want_grad):
    """K and, when asked, dK/dx and dK/dnu, in slabs of pairs."""
    outs = [torch.empty_like(x) for _ in range(3 if want_grad else 1)]
    t, w = _nodes(1e-3)
    ch = torch.cosh(t)
    for i in range(0, x.numel(), 200000):
        xi, vi = x[i:i + 200000, None], nu[i:i + 200000, None]
        e = vi * t - xi * ch + torch.log(w)
        top = e.max(dim=1, keepdim=True).values
        f = torch.exp(e - top)
        back = torch.exp(-2 * vi * t)
        scale = 0.5 * torch.exp(top[:, 0])
        outs[0][i:i + 200000] = scale * (f * (1 + back)).sum(1)
        if want_grad:
            outs[1][i:i + 200000] = -scale * (f * (1 + back) * ch).sum(1)
            outs[2][i:i + 200000] = scale * (f * (1 - back) * t).sum(1)
    return outs


def exact(case, seed):
    kind, dt = case["kind"], torch.float64
    if kind in ("matern", "host"):
        n = case["n"]
        if n > 20000 and case["nu"] not in (0.5, 1.5, 2.5):
            return None  # over 20 seconds
        L = _locs(n, seed)
        out = _matrix(L, L, case["beta"], case["nu"], 1.0, dt)
        return out.cpu() if kind == "host" else out
    if kind == "cross":
        return _matrix(_locs(case["m"], seed), torch.as_tensor(_targets(case, seed), device="cuda"),
                       case["beta"], case["nu"], 1.0, dt)
    if kind == "batched":
        outs = []
        for i in _instances(case, seed):
            L = torch.as_tensor(i.locations(), device="cuda")
            outs.append(_matrix(L, L, i.beta, i.nu, i.sigma2, dt))
        return outs
    if kind == "eval":
        k = _pair_sums(*_pairs(case, seed), False)[0]
        if case["form"] != "f64":
            k = torch.where(k.float().isinf(), math.inf, k)
        return k
    if kind == "grad":
        return tuple(_pair_sums(*_pairs(case, seed), True))
    L = _locs(case["n"], seed)
    m = _matrix(L, L, case["beta"], case["nu"], 1.0, dt)
    z = _observations(case, L, seed)
    f = torch.linalg.cholesky(m)
    y = torch.linalg.solve_triangular(f, z[:, None], upper=False)[:, 0]
    logdet, q = 2 * f.diagonal().log().sum(), (y * y).sum()
    out = torch.stack([-0.5 * (q + logdet + case["n"] * math.log(2 * math.pi)), logdet, q])
    # the factor below the diagonal of the column-major matrix, the matrix above it
    return {"out": out, "a": f.T.contiguous().triu_() + m.tril_(-1), "y": y}
