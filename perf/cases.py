"""The workloads whose speed is tracked: whole solves, repeated evaluations on
a kept plan, batched evaluation and the direct sum, each through the public
entry points of paper_2002_04894_gb300 as a user's program calls them.

A case is a dict:
  form      solve   fmm_plan + fmm_eval + fmm_destroy on device arrays
            host    the same on host arrays (what the server does per request)
            eval    fmm_eval with the charges at hand on a plan kept by the caller
            batch   fmm_batch_launch over many kept plans
            direct  fmm_direct, the exact sum at sampled targets
  kind      point distribution;  n  points (batch: the largest system)
  levels, p, theta, prec ("mixed" or "fp64"), tight, eta, step (bisections per
  expansion level), fields: the plan's and evaluation's options
Mixed-form cases take float32 points and charges, plain-form ones float64.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2002_04894_gb300 as fmm


def _case(name, form, kind, n, levels, p, prec="mixed", tight=False, eta=1.0, step=1, fields=True, theta=0.5,
          systems=0, targets=0):
    c = dict(form=form, kind=kind, n=n, levels=levels, p=p, theta=theta, prec=prec, tight=tight, eta=eta,
             step=step, fields=fields, systems=systems, targets=targets)
    return dict(c, name=name) if name else c


def _levels(n, leaf=100.0):
    """Binary levels for about `leaf` points per leaf (the server's policy)."""
    return max(0, int(round(math.log2(max(n, 1) / leaf))))


def listed():
    return [
        # the smallest request a server sees: host arrays in and out, a handful of leaves; latency only
        _case("host_1k", "host", "uniform", 1000, 3, 8),
        # a small system whose plan is kept, potential only (a time step's energy)
        _case("eval_5k_potential", "eval", "plummer", 5003, 6, 8, fields=False),
        # the small uniform configuration in plain double precision, evaluated again with new charges
        _case("eval_20k_fp64", "eval", "uniform", 20_000, 8, 8, prec="fp64"),
        # the parameter study: 100,000 points, octree levels, splits between median and midpoint
        _case("octree_100k", "solve", "gaussian", 100_000, 12, 12, eta=0.5, step=3),
        # a large served request: clustered points on the host, odd size
        _case("host_300k", "host", "plummer", 300_007, 12, 10),
        # a big plain double-precision evaluation (the accuracy anchor of the method)
        _case("eval_200k_fp64", "eval", "plummer", 200_000, 11, 10, prec="fp64"),
        # many independent systems of very different sizes, all evaluations in one launch
        _case("batch_48", "batch", "uniform", 200_000, 0, 12, systems=48),
        # iterative use: new charges on a kept plan of a strongly clustered set, odd size
        _case("eval_1m", "eval", "gmm", 1_000_003, 14, 12, tight=True),
        # the exact sum at sampled targets, which users check accuracy with
        _case("direct_500k", "direct", "plummer", 500_000, 0, 0, targets=1000),
        # 2M clustered points, cell boxes, one solve per time step
        _case("solve_2m", "solve", "plummer", 2_000_000, 14, 12),
        # multiscale disc, octree levels, eta-weighted splits (the galaxy experiment)
        _case("galaxy_2m", "solve", "galaxy", 2_000_000, 15, 12, eta=0.625, step=3),
        # the headline solve: 8M points of a Gaussian mixture, tight boxes
        _case("solve_8m", "solve", "gmm", 8_000_000, 17, 12, tight=True),
    ]


def draw(rng):
    form = rng.choice(["solve", "solve", "solve", "host", "eval", "eval", "fp64", "octree", "batch", "direct"])

    def size(lo, hi):
        return int(math.exp(rng.uniform(math.log(lo), math.log(hi)))) | 1

    leaf = rng.uniform(50.0, 150.0)
    p = rng.choice([6, 8, 9, 10, 11, 12])
    if form == "fp64":
        n = size(1000, 150_000)
        return _case(None, rng.choice(["solve", "eval"]), rng.choice(["uniform", "plummer"]), n, _levels(n, leaf),
                     rng.choice([6, 8, 10]), prec="fp64")
    if form == "octree":
        n = size(3000, 1_000_000)
        return _case(None, "solve", rng.choice(["uniform", "plummer", "gaussian", "galaxy"]), n,
                     3 * max(1, round(_levels(n, leaf) / 3)), p, eta=rng.choice([0.5, 0.625, 0.75, 1.0]), step=3)
    if form == "batch":
        return _case(None, "batch", "uniform", size(20_000, 200_000), 0, rng.choice([8, 10, 12]),
                     systems=rng.randrange(8, 49))
    if form == "direct":
        return _case(None, "direct", rng.choice(["uniform", "plummer"]), size(2000, 1_000_000), 0, 0,
                     targets=rng.randrange(1, 1001))
    n = size(1000, {"solve": 4_000_000, "host": 1_000_000, "eval": 4_000_000}[form])
    kind = rng.choice(["uniform", "plummer", "gmm"])
    return _case(None, form, kind, n, _levels(n, leaf), p, tight=kind == "gmm" or rng.random() < 0.3,
                 fields=rng.random() < 0.8)


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _isotropic(n, g):
    v = torch.randn((n, 3), generator=g, device="cuda", dtype=torch.float64)
    return v / v.norm(dim=1, keepdim=True)


def _points(kind, n, g):
    """n x 3 float64 points on the device: the distributions of the package's inputs module."""
    f64 = dict(generator=g, device="cuda", dtype=torch.float64)
    if kind == "uniform":
        return torch.rand((n, 3), **f64)
    if kind == "gaussian":
        return 0.5 + 0.1 * torch.randn((n, 3), **f64)
    if kind == "plummer":  # scale radius 0.1, truncated at ten times that: radii by inversion on the kept mass
        top = (1.0 + 0.01) ** -1.5
        u = torch.rand(n, **f64) * (top * (1 - 1e-12)) + 1e-14
        return 0.5 + (0.1 / (u ** (-2.0 / 3.0) - 1.0).sqrt())[:, None] * _isotropic(n, g)
    if kind == "gmm":  # 16 components, centres uniform, sigma log-uniform in [1e-3, 1e-1]
        centres = torch.rand((16, 3), **f64)
        sigma = 10.0 ** (2.0 * torch.rand(16, **f64) - 3.0)
        k = torch.randint(0, 16, (n,), generator=g, device="cuda")
        return centres[k] + sigma[k, None] * torch.randn((n, 3), **f64)
    if kind == "galaxy":  # a two-armed ring, refined in generations of ten points in shrinking flat spheroids
        m = min(10_000, n)
        r = 6000.0 + 12000.0 * torch.rand(m, **f64)
        arm = torch.randint(0, 2, (m,), generator=g, device="cuda")
        phi = torch.log(r / 6000.0) / math.tan(math.radians(15.0)) + math.pi * arm + 0.1 * torch.randn(m, **f64)
        x = torch.stack([r * phi.cos(), r * phi.sin(), 300.0 * torch.randn(m, **f64)], 1)
        big = 900.0
        while len(x) < n:
            need = min(n, 10 * len(x))
            parents = x[torch.randperm(len(x), generator=g, device="cuda")][: -(-need // 10)]
            off = _isotropic(need, g) * torch.rand(need, **f64)[:, None] ** (1.0 / 3.0)
            x = parents.repeat_interleave(10, 0)[:need] + off * torch.tensor([big, big, big / 10.0], device="cuda",
                                                                             dtype=torch.float64)
            big *= 2.0 / 3.0
        return 0.5 + x / 39600.0
    raise ValueError(kind)


def _dtype(case):
    return torch.float64 if case["prec"] == "fp64" else torch.float32


def _inputs(case, seed):
    """Points and charges of one system: charges uniform in [-1, 1), or +-1 for the Gaussian mixture."""
    g = _gen(seed)
    x = _points(case["kind"], case["n"], g).to(_dtype(case)).contiguous()
    q = 2.0 * torch.rand(case["n"], generator=g, device="cuda", dtype=torch.float64) - 1.0
    q = torch.where(q < 0, -1.0, 1.0) if case["kind"] == "gmm" else q
    return x, q.to(_dtype(case)).contiguous()


def _batch_inputs(case, seed):
    """Sizes log-uniform up to n, uniform and Plummer alternating. The sizes belong to the case, the points to the seed."""
    sizes = np.random.default_rng([case["systems"], case["n"]])
    ns = np.exp(sizes.uniform(np.log(1e3), np.log(case["n"]), case["systems"])).astype(int)
    return [_inputs(dict(case, n=int(n), kind=("uniform", "plummer")[i % 2]), seed * 1000 + i) for i, n in enumerate(ns)]


def _plan(case, x):
    prec = fmm.FMM_PREC_FP64 if case["prec"] == "fp64" else fmm.FMM_PREC_MIXED
    return fmm.fmm_plan(x, case["levels"], case["p"], case["theta"], prec=prec, eta=case["eta"],
                        bisections_per_level=case["step"], tight=case["tight"])


def prepare(case, seed):
    form = case["form"]
    if form == "batch":
        xq = _batch_inputs(case, seed)
        plans = [_plan(dict(case, levels=_levels(len(q))), x) for x, q in xq]
        ends = np.cumsum([0] + [len(q) for _, q in xq])
        pot = torch.empty(int(ends[-1]), dtype=torch.float32, device="cuda")
        fld = torch.empty((int(ends[-1]), 3), dtype=torch.float32, device="cuda")
        cut = list(zip(ends[:-1], ends[1:]))
        batch = fmm.fmm_batch_create(plans, [q for _, q in xq], [pot[a:b] for a, b in cut], [fld[a:b] for a, b in cut])
        return dict(case=case, batch=batch, pot=pot, fld=fld)
    x, q = _inputs(case, seed)
    s = dict(case=case, x=x, q=q)
    if form == "host":
        s["x"], s["q"] = x.cpu().numpy(), q.cpu().numpy()
    elif form == "eval":
        s["plan"] = _plan(case, x)
    elif form == "direct":
        s["targets"] = torch.randperm(case["n"], generator=_gen(seed + 1), device="cuda")[: case["targets"]].sort()[0]
    return s


def run(state):
    case, form = state["case"], state["case"]["form"]
    if form == "batch":
        fmm.fmm_batch_launch(state["batch"])
        return state["pot"], state["fld"]
    if form == "direct":
        return fmm.fmm_direct(state["x"], state["q"], state["targets"])
    if form == "eval":
        return fmm.fmm_eval(state["plan"], state["q"], want_fields=case["fields"])
    plan = _plan(case, state["x"])
    out = fmm.fmm_eval(plan, state["q"], want_fields=case["fields"])
    fmm.fmm_destroy(plan)
    return out


def work(case):
    """Bytes: points (where the plan is part of the call) and charges in, results out. Flops: 20 per near pair and
    12 sum (n + 1)^2 per M2L pair (the rotational form), with the list lengths that theta = 0.5 gives in the bulk of
    these distributions (about 150 near leaves and 800 M2L pairs per leaf), bounded by the number of leaves."""
    size = 8 if case["prec"] == "fp64" else 4
    if case["form"] == "direct":
        t = min(case["targets"], case["n"])
        return {"bytes": size * (4 * case["n"] + 4 * t) + 8 * t, "flops": 20.0 * t * case["n"]}
    if case["form"] == "batch":
        sizes = np.random.default_rng([case["systems"], case["n"]])
        ns = np.exp(sizes.uniform(np.log(1e3), np.log(case["n"]), case["systems"])).astype(int)
        each = [work(dict(case, form="eval", n=int(n), levels=_levels(int(n)))) for n in ns]
        return {k: float(sum(w[k] for w in each)) for k in ("bytes", "flops")}
    n, leaves = case["n"], 1 << case["levels"]
    words = n * (1 + 1 + (3 if case["fields"] else 0) + (0 if case["form"] == "eval" else 3))
    near = n * (n / leaves) * min(150, leaves)
    m2l = leaves * min(800, leaves // 2) * sum((k + 1) ** 2 for k in range(case["p"] + 1))
    return {"bytes": float(size * words), "flops": 20.0 * near + 12.0 * m2l}


def _direct(x, q, targets=None):
    """Potential and field of every target by the direct sum in double precision, pairs at zero distance skipped."""
    x, q = x.double(), q.double()
    t = x if targets is None else x[targets]
    pot = torch.empty(len(t), dtype=torch.float64, device=x.device)
    fld = torch.empty((len(t), 3), dtype=torch.float64, device=x.device)
    step = max(1, (1 << 21) // len(x))
    cols = [x[:, a].contiguous() for a in range(3)]
    for i in range(0, len(t), step):
        d = [t[i:i + step, a, None] - cols[a] for a in range(3)]
        r2 = d[0] * d[0]
        r2.addcmul_(d[1], d[1]).addcmul_(d[2], d[2])
        w = r2.rsqrt_()
        w.masked_fill_(torch.isinf(w), 0.0)
        qr = w * q
        pot[i:i + step] = qr.sum(1)
        qr.mul_(w).mul_(w)
        for a in range(3):
            fld[i:i + step, a] = d[a].mul_(qr).sum(1)
    return pot, fld


def exact(case, seed):
    if case["form"] == "batch":
        xq = _batch_inputs(case, seed)
        if sum(len(q) ** 2 for _, q in xq) > 6e10:
            return None
        each = [_direct(x, q) for x, q in xq]
        return torch.cat([e[0] for e in each]), torch.cat([e[1] for e in each])
    if case["form"] == "direct":
        x, q = _inputs(case, seed)
        t = torch.randperm(case["n"], generator=_gen(seed + 1), device="cuda")[: case["targets"]].sort()[0]
        return _direct(x, q, t)
    if case["n"] > 210_000:
        return None
    pot, fld = _direct(*_inputs(case, seed))
    return pot, (fld if case["fields"] else None)
