"""The calls whose speed is followed: what a user of the magnitude solver has it
do, through the Python package's entry points, from one small solve to the
100,000-point benchmark step.

A case is a dict of plain values.  ``kind`` names the entry point, ``cloud``
the distribution of the points (the clouds of ``workloads.py``, drawn on the
GPU from a seed), ``n`` x ``m`` their size and ``t`` the scale.  All calls go
through the package's cached context of the current stream, as ``mag.solve``
and ``mag.magnitude`` do, so its workspace is kept between calls.
"""
from __future__ import annotations

import math

import torch

import paper_2607_23354_gb300 as mag

# Scales: the t of a case is where the weighting is used in earnest -- between
# strongly coupled points and the bound log(n-1)/min d, past which Z is nearly I.


def listed():
    return [
        # one small space, the package's smoke size: launches and waits are all of it
        dict(name="solve_small", kind="solve", cloud="cube", n=300, m=8, t=1.0),
        # the precision tables' cloud: a dense solve of middle size in R^3
        dict(name="solve_mixture", kind="solve", cloud="mixture", n=16384, m=3, t=5.0),
        # the paper's high-dimensional runtime configuration
        dict(name="solve_highdim", kind="solve", cloud="normal", n=10000, m=100, t=0.5),
        # the headline benchmark step: three scales on 1e5 points, the bound found inside
        dict(name="multi_headline", kind="multi", cloud="cube", n=100000, m=8, t=1.0, t2=10.0),
        # the paper's task: the cutoff t_+ by bisection from 1e-3, N(0, I_10)
        dict(name="sweep_paper", kind="sweep", cloud="normal", n=3000, m=10, t=1e-3, method="bisection"),
        # a training step: weighting forward, the gradients of a loss of w backward
        dict(name="grad_adjoint", kind="grad", cloud="normal16", n=8192, m=16, t=2.0),
        # many small spaces of uneven size at several scales in one call
        dict(name="batch_uneven", kind="batch", cloud="normal", n=2048, n_min=64, m=32, t=0.1, t2=10.0,
             clouds=256, nt=4),
        # one weighting of a third of the benchmark's points, the parity tests' larger cloud
        dict(name="solve_cube", kind="solve", cloud="cube", n=32768, m=8, t=10.0),
        # checking a weighting that came from elsewhere: the FP64 residual
        dict(name="residual_check", kind="residual", cloud="cube", n=30000, m=8, t=2.0),
        # the bound on t_+ alone, at the paper's largest size
        dict(name="min_distance", kind="min_distance", cloud="normal", n=30000, m=10, t=0.0),
        # the similarity matrix itself, dense FP64
        dict(name="similarity", kind="similarity", cloud="mixture", n=8192, m=3, t=1.0, precision="fp64"),
        # the plain dense method's factor: FP64 Cholesky, ragged size
        dict(name="factor_fp64", kind="factor", cloud="normal", n=5001, m=10, t=1.0, precision="fp64"),
    ]


def _log_int(rng, lo, hi):
    """A size spread over the logarithm of its range; odd and ragged ones as they fall."""
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["solve", "solve", "solve", "multi", "sweep", "grad", "batch", "residual", "min_distance",
                       "similarity", "factor"])
    c = dict(kind=kind)
    if kind == "solve":
        cloud = rng.choice(["cube", "mixture", "normal"])
        m = {"cube": rng.randint(6, 16), "mixture": 3, "normal": rng.choice([10, 30, 100, rng.randint(10, 120)])}[cloud]
        t = {"cube": rng.uniform(6.0, 25.0), "mixture": rng.uniform(5.0, 20.0),
             "normal": rng.uniform(2.0, 6.0) if m < 30 else rng.uniform(0.5, 3.0)}[cloud]
        c.update(cloud=cloud, n=_log_int(rng, 60, 40000), m=m, t=t)
    elif kind == "multi":
        c.update(cloud="cube", n=_log_int(rng, 500, 60000), m=rng.randint(8, 12), t=rng.uniform(4.0, 8.0),
                 t2=rng.uniform(10.0, 30.0))
    elif kind == "sweep":
        c.update(cloud=rng.choice(["normal", "halving"]), n=_log_int(rng, 500, 6000), m=rng.choice([3, 10, 30, 100]),
                 t=1e-3, method=rng.choice(["bisection", "ridders"]))
    elif kind == "grad":
        c.update(cloud="normal16", n=_log_int(rng, 300, 12000), m=rng.randint(8, 38), t=rng.uniform(2.0, 8.0))
    elif kind == "batch":
        n_min = _log_int(rng, 16, 256)
        c.update(cloud="normal", n=_log_int(rng, 300, 2048), n_min=n_min, m=rng.randint(16, 48), t=rng.uniform(0.1, 1.0),
                 t2=rng.uniform(2.0, 10.0), clouds=rng.randint(8, 300), nt=rng.randint(1, 4))
    elif kind == "residual":
        c.update(cloud=rng.choice(["cube", "normal16"]), n=_log_int(rng, 200, 40000), m=rng.randint(2, 38),
                 t=rng.uniform(0.5, 8.0))
    elif kind == "min_distance":
        c.update(cloud=rng.choice(["cube", "mixture", "normal", "halving"]), n=_log_int(rng, 200, 60000),
                 m=rng.choice([3, 10, 30, rng.randint(2, 64)]), t=0.0)
        if c["cloud"] == "mixture":
            c["m"] = 3
    elif kind == "similarity":
        c.update(cloud=rng.choice(["cube", "mixture", "normal"]), n=_log_int(rng, 200, 12000), m=rng.randint(2, 40),
                 t=rng.uniform(0.5, 8.0), precision=rng.choice(["fp64", "fp64", "fp32"]))
        if c["cloud"] == "mixture":
            c["m"] = 3
    else:
        c.update(cloud=rng.choice(["cube", "normal"]), n=_log_int(rng, 200, 6000), m=rng.randint(6, 20),
                 t=rng.uniform(1.0, 6.0), precision=rng.choice(["fp64", "fp64", "fp16x3"]))
    return c


def _points(cloud, n, m, g):
    if cloud == "cube":  # uniform in [0, 1]^m
        return torch.rand(n, m, generator=g, dtype=torch.float64, device="cuda")
    x = torch.randn(n, m, generator=g, dtype=torch.float64, device="cuda")
    if cloud == "normal":  # N(0, I)
        return x
    if cloud == "normal16":  # N(0, I / m): unit spread whatever m, the gradient workload's cloud
        return x / math.sqrt(m)
    if cloud == "halving":  # N(0, Sigma), Sigma_jj = 2^-(j-1)
        return x * torch.sqrt(2.0 ** -torch.arange(m, dtype=torch.float64, device="cuda"))
    # mixture: 8 isotropic components, means uniform in [0, 10]^m, sigma 0.5
    means = 10.0 * torch.rand(8, m, generator=g, dtype=torch.float64, device="cuda")
    comp = torch.randint(0, 8, (n,), generator=g, device="cuda")
    return means[comp] + 0.5 * x


def _batch_sizes(case):
    lo, hi, k = min(case["n_min"], case["n"]), case["n"], case["clouds"]
    return [max(2, int(round(lo * (hi / lo) ** ((i + 0.5) / k)))) for i in range(k)]


def _batch_ts(case):
    k = case["nt"]
    return [case["t"]] if k == 1 else [case["t"] * (case["t2"] / case["t"]) ** (i / (k - 1)) for i in range(k)]


def prepare(case, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    kind = case["kind"]
    s = dict(case=case)
    if kind == "batch":
        sizes = _batch_sizes(case)
        x = _points(case["cloud"], sum(sizes), case["m"], g)
        s["clouds"] = [c.clone() for c in x.split(sizes)]
        s["ts"] = _batch_ts(case)
        return s
    s["X"] = _points(case["cloud"], case["n"], case["m"], g)
    if kind == "grad":  # leaves of a training step, and the loss's dL/dw
        s["X"].requires_grad_()
        s["t"] = torch.tensor(case["t"], dtype=torch.float64, device="cuda", requires_grad=True)
        s["c"] = torch.rand(case["n"], generator=g, dtype=torch.float64, device="cuda")
    if kind == "residual":  # an approximate weighting
        e = torch.randn(case["n"], generator=g, dtype=torch.float64, device="cuda")
        s["w"] = (1.0 + 0.2 * e) / math.sqrt(case["n"])
    return s


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind == "solve":
        w, M = mag.solve(state["X"], case["t"])
        return w, M
    if kind == "grad":
        w, M = mag.magnitude(state["X"], state["t"])
        dX, dt = torch.autograd.grad((state["c"] * w).sum(), (state["X"], state["t"]))
        return w.detach(), M.detach(), dX, dt
    if kind == "sweep":
        r = mag.sweep_tplus(state["X"], t_lo=case["t"], method=case["method"])
        return torch.tensor([r["t_plus"], *r["bracket"], r["mag"]], dtype=torch.float64), r["w"]
    ctx = mag.default_context()
    if kind == "multi":
        W, Ms, _ = ctx.solve_multi(state["X"], [case["t"], case["t2"], "bound"])
        return W, torch.tensor(Ms, dtype=torch.float64)
    if kind == "batch":
        ws, M, st = ctx.solve_batch(state["clouds"], state["ts"])
        return torch.cat(ws), M, st
    if kind == "residual":
        r, norms = ctx.residual(state["X"], case["t"], state["w"])
        return r, torch.tensor([norms["rel_residual"], norms["r_norm_inf"], norms["z_norm_inf"],
                                norms["w_norm_inf"]], dtype=torch.float64)
    if kind == "min_distance":
        return torch.tensor(ctx.min_distance(state["X"]), dtype=torch.float64)
    if kind == "similarity":
        return ctx.similarity_matrix(state["X"], case["t"], case["precision"])
    return ctx.cholesky_factor(state["X"], case["t"], case["precision"])


def work(case):
    """Each input read once, each output written once; the operations of the
    definition: 3 m + 2 per pair for its distance and entry, n^3/3 per factor,
    4 n^2 per right-hand side's sweeps and residual."""
    n, m, kind = float(case["n"]), float(case["m"]), case["kind"]
    pairs = n * (n - 1) / 2 * (3 * m + 2)
    solve = n**3 / 3 + 4 * n * n
    points = 8 * n * m
    if kind == "solve":
        return dict(bytes=points + 8 * n, flops=pairs + solve)
    if kind == "multi":
        return dict(bytes=points + 24 * n, flops=pairs + 3 * solve)
    if kind == "sweep":  # the two ends and one solve per halving to 1e-6
        return dict(bytes=points + 8 * n, flops=pairs + 22 * solve)
    if kind == "grad":  # forward, the adjoint's sweeps, the gradient over the pairs
        return dict(bytes=2 * points + 16 * n, flops=2 * pairs + solve + 4 * n * n)
    if kind == "batch":
        k = case["nt"]
        sizes = [float(v) for v in _batch_sizes(case)]
        return dict(bytes=sum(8 * v * m + 8 * v * k for v in sizes),
                    flops=sum(v * v / 2 * (3 * m + 2) + k * (v**3 / 3 + 4 * v * v) for v in sizes))
    if kind == "residual":
        return dict(bytes=points + 16 * n, flops=pairs + 2 * n * n)
    if kind == "min_distance":
        return dict(bytes=points, flops=pairs)
    out = n * n * (8 if case["precision"] == "fp64" else 4)
    if kind == "similarity":
        return dict(bytes=points + out, flops=pairs)
    return dict(bytes=points + out, flops=pairs + n**3 / 3)


def _dist(X):
    return torch.cdist(X, X, compute_mode="donot_use_mm_for_euclid_dist")


def _sym_solve(Z, B):
    """Z^{-1} B in FP64 by Cholesky (LU when Z is not positive definite to rounding), one refinement step."""
    L, info = torch.linalg.cholesky_ex(Z)
    if int(info) == 0:
        x = torch.cholesky_solve(B, L)
        return x + torch.cholesky_solve(B - Z @ x, L)
    LU, piv = torch.linalg.lu_factor(Z)
    x = torch.linalg.lu_solve(LU, piv, B)
    return x + torch.linalg.lu_solve(LU, piv, B - Z @ x)


def _weighting(d, t):
    one = torch.ones(d.shape[0], 1, dtype=torch.float64, device=d.device)
    return _sym_solve(torch.exp(-t * d), one)[:, 0]


def _sweep(X, t_lo, method, rel_tol=1e-6):
    d = _dist(X)
    n = X.shape[0]
    off = d.clone()
    off.fill_diagonal_(math.inf)
    lo, hi = t_lo, math.log(n - 1) / float(off.min())
    del off
    best = {}

    def f(t):
        w = _weighting(d, t)
        v = float(w.min())
        if v >= 0:
            best["w"] = w
        return v

    fhi, flo = f(hi), f(lo)
    if flo >= 0:
        w = best["w"]
        return [lo, lo, lo, float(w.sum())], w
    prev = math.nan
    while hi - lo > rel_tol * hi:
        x1, f1, f2 = lo, flo, fhi
        x3 = lo + (hi - lo) / 2

        def move(x):
            nonlocal lo, hi, flo, fhi
            v = f(x)
            if v >= 0:
                hi, fhi = x, v
            else:
                lo, flo = x, v
            return v

        f3 = move(x3)
        if method == "bisection" or hi - lo <= rel_tol * hi:
            continue
        sq = math.sqrt(f3 * f3 - f1 * f2)
        if not sq > 0:
            continue
        x4 = x3 + (x3 - x1) * (1.0 if f1 >= f2 else -1.0) * f3 / sq
        if not lo < x4 < hi:
            prev = math.nan
            continue
        move(x4)
        if hi - lo <= rel_tol * hi:
            break
        delta = 0.5 * rel_tol * hi
        if abs(x4 - prev) <= delta:
            xc = x4 - delta if hi == x4 else x4 + delta
            if lo < xc < hi:
                move(xc)
        prev = x4
    w = best["w"]
    return [hi, lo, hi, float(w.sum())], w


def exact(case, seed):
    kind, n = case["kind"], case["n"]
    if kind == "multi" and n > 16384 or kind == "solve" and n > 20000:
        return None  # an FP64 factor of this size takes too long
    s = prepare(case, seed)
    if kind == "batch":
        ws, Ms = [], []
        for x in s["clouds"]:
            d = _dist(x)
            for t in s["ts"]:
                w = _weighting(d, t)
                ws.append(w)
                Ms.append(w.sum())
        M = torch.stack(Ms).reshape(len(s["clouds"]), len(s["ts"]))
        return torch.cat(ws), M, torch.zeros(M.shape, dtype=torch.int32)
    X = s["X"].detach()
    if kind in ("residual", "min_distance"):
        rows = []
        zmax, dmin = 0.0, math.inf
        for i in range(0, n, 2048):
            d = torch.cdist(X[i:i + 2048], X, compute_mode="donot_use_mm_for_euclid_dist")
            if kind == "min_distance":
                d.diagonal(i).fill_(math.inf)
                dmin = min(dmin, float(d.min()))
            else:
                Z = torch.exp(-case["t"] * d)
                zmax = max(zmax, float(Z.sum(1).max()))
                rows.append(1.0 - Z @ s["w"])
        if kind == "min_distance":
            return torch.tensor([dmin, math.log(n - 1) / dmin], dtype=torch.float64)
        r = torch.cat(rows)
        rn, wn = float(r.abs().max()), float(s["w"].abs().max())
        return r, torch.tensor([rn / (zmax * wn), rn, zmax, wn], dtype=torch.float64)
    if kind == "sweep":
        v, w = _sweep(X, case["t"], case["method"])
        return torch.tensor(v, dtype=torch.float64), w
    d = _dist(X)
    if kind == "solve":
        w = _weighting(d, case["t"])
        return w, float(w.sum())
    if kind == "multi":
        off = d.clone()
        off.fill_diagonal_(math.inf)
        W = torch.stack([_weighting(d, t) for t in (case["t"], case["t2"], math.log(n - 1) / float(off.min()))])
        return W, W.sum(1).cpu()
    t = case["t"]
    Z = torch.exp(-t * d)
    if kind == "similarity":
        return Z
    if kind == "factor":
        return torch.linalg.cholesky(Z)
    # grad: lambda = Z^{-1} c, dL/dt = lambda^T (d o Z) w, dL/dx_i = t sum_k G_ik (x_i - x_k)
    x = _sym_solve(Z, torch.stack([torch.ones_like(s["c"]), s["c"]], 1))
    w, lam = x[:, 0], x[:, 1]
    dt = lam @ ((d * Z) @ w)
    d.fill_diagonal_(1.0)
    G = Z / d * (torch.outer(lam, w) + torch.outer(w, lam))
    G.fill_diagonal_(0.0)
    dX = t * (X * G.sum(1, keepdim=True) - G @ X)
    return w, w.sum(), dX, dt
