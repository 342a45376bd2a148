"""The work that users of the solver have it do, as timed cases over its public entry points.

``listed()`` names the cases, ``draw(rng)`` gives more of the same ranges, ``prepare`` makes
what a program holds before the call (tensors on the GPU, or page-locked host arrays where
the call takes host batches), ``run`` makes one pass, ``work`` counts what a pass cannot do
without and ``exact`` gives the results in 64 bits from plain torch.

Distributions are those of the benchmark and the tests: type-1 LPs ``A ~ U[0.1, 1]``,
``b ~ U[1, 10]``, ``c ~ U[0, 1]`` (slack basis feasible); type-2 LPs built around a point
``x0 ~ U[0, 1]^n`` with half of the rows ``>=`` (slack basis infeasible, about 5% infeasible
and 5% unbounded); boxes ``l ~ U[-10, 0]``, ``u ~ U[0, 10]``, ``c ~ N(0, 1)``.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_1609_08114_gb300 import LPBatch, Solver, solve

DTYPES = {"f32": torch.float32, "f64": torch.float64}
_solver = None


def listed():
    return [
        # One control step's worth of small LPs: the call where launches and the host path count.
        dict(name="small_1000x16", kind="dense", count=1000, m=16, n=16, dtype="f64", prec="fp32_refine", rule="lpc"),
        # The smallest LPs of the size sweep, in the number that fills the GPU.
        dict(name="tiny_100000x5", kind="dense", count=100_000, m=5, n=5, dtype="f64", prec="fp32_refine", rule="lpc"),
        # FP32 data of an odd shape, as features from an FP32 pipeline come.
        dict(name="f32_30000x48x37", kind="dense", count=30_000, m=48, n=37, dtype="f32", prec="fp32_refine", rule="lpc"),
        # The benchmark's headline batch.
        dict(name="hundred_50000x100", kind="dense", count=50_000, m=100, n=100, dtype="f64", prec="fp32_refine",
             rule="lpc"),
        # The plain FP64 tableau that the benchmark compares it with.
        dict(name="plain64_20000x100", kind="dense", count=20_000, m=100, n=100, dtype="f64", prec="fp64", rule="lpc"),
        # The top of the size sweep: LPs whose tableau does not fit an SM's shared memory.
        dict(name="large_2000x300", kind="dense", count=2000, m=300, n=300, dtype="f64", prec="fp32_refine", rule="lpc"),
        # Infeasible starts: Phase I, infeasible and unbounded LPs, the FP64 re-solve.
        dict(name="twophase_4000x200", kind="twophase", count=4000, m=200, n=200, prec="fp32_refine", rule="lpc"),
        # An LP layer in training on LPs of mixed sizes: forward, then the gradients of A, b and c.
        dict(name="grad_mixed_6000", kind="grad", count=6000, lo=8, hi=256, dtype="f64"),
        # The support function of one polytope in many directions (reachability).
        dict(name="shared_50000x100", kind="shared", count=50_000, m=100, n=100, dtype="f64", prec="fp32_refine",
             sweep=False),
        # Variables with bounds l <= x <= u.
        dict(name="bounded_10000x100", kind="bounded", count=10_000, m=100, n=100, prec="fp32_refine"),
        # Support functions of boxes, the closed form.
        dict(name="box64_3000000x28", kind="box", count=3_000_000, n=28, dtype="f64", one_box=False),
        # A batch and results in host memory, through the copy / solve / copy-back pipeline.
        dict(name="host_10000x100", kind="host", count=10_000, m=100, n=100, prec="fp32_refine"),
    ]


def _log(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["dense"] * 6 + ["twophase", "twophase", "grad", "grad", "shared", "bounded", "box", "box", "host"])
    if kind == "dense":
        prec = rng.choice(["fp32_refine"] * 4 + ["fp64", "fp64", "fp32"])
        m, n = _log(rng, 4, 300), _log(rng, 4, 300)
        most = min(120_000, (500_000_000 if prec != "fp64" else 200_000_000) // (m * n))
        return dict(kind=kind, count=_log(rng, 500, max(600, most)), m=m, n=n, dtype=rng.choice(["f64", "f64", "f32"]),
                    prec=prec, rule=rng.choice(["lpc"] * 5 + ["rpc"]))
    if kind == "twophase":
        m, n = _log(rng, 10, 200), _log(rng, 10, 200)
        return dict(kind=kind, count=_log(rng, 300, min(6000, 120_000_000 // (m * n))), m=m, n=n,
                    prec=rng.choice(["fp32_refine"] * 3 + ["fp64"]) if m * n <= 6000 else "fp32_refine",
                    rule=rng.choice(["lpc", "lpc", "steepest"]))
    if kind == "grad":
        lo = rng.randint(4, 40)
        return dict(kind=kind, count=_log(rng, 500, 6000), lo=lo, hi=_log(rng, lo + 8, 256),
                    dtype=rng.choice(["f64", "f64", "f32"]))
    if kind == "shared":
        return dict(kind=kind, count=_log(rng, 1000, 50_000), m=_log(rng, 10, 100), n=_log(rng, 10, 100),
                    dtype=rng.choice(["f64", "f32"]), prec="fp32_refine", sweep=rng.random() < 0.5)
    if kind == "bounded":
        return dict(kind=kind, count=_log(rng, 500, 10_000), m=_log(rng, 8, 100), n=_log(rng, 8, 100),
                    prec=rng.choice(["fp32_refine", "fp32_refine", "fp64"]))
    if kind == "box":
        n = _log(rng, 3, 60)
        return dict(kind=kind, count=_log(rng, 10_000, min(6_000_000, 84_000_000 // n)), n=n,
                    dtype=rng.choice(["f32", "f64"]), one_box=rng.random() < 0.3)
    return dict(kind=kind, count=_log(rng, 1000, 10_000), m=_log(rng, 20, 100), n=_log(rng, 20, 100),
                prec="fp32_refine")


# ---- inputs -----------------------------------------------------------------

def _solver_():
    global _solver
    if _solver is None:
        _solver = Solver(0)
    return _solver


def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _uniform(g, shape, lo, hi, dtype=torch.float64):
    return torch.rand(shape, generator=g, device="cuda", dtype=dtype).mul_(hi - lo).add_(lo)


def _type1(case, seed):
    g, dt = _gen(seed), DTYPES[case.get("dtype", "f64")]
    k, m, n = case["count"], case["m"], case["n"]
    return _uniform(g, (k, m, n), 0.1, 1.0, dt), _uniform(g, (k, m), 1.0, 10.0, dt), _uniform(g, (k, n), 0.0, 1.0, dt)


def _type2(case, seed):
    g = _gen(seed)
    k, m, n = case["count"], case["m"], case["n"]
    half = m // 2
    x0, A, c = _uniform(g, (k, n), 0.0, 1.0), _uniform(g, (k, m, n), 0.1, 1.0), _uniform(g, (k, n), 0.0, 1.0)
    sel = _uniform(g, (k,), 0.0, 1.0)
    inf, unb = torch.nonzero(sel < 0.05)[:, 0], torch.nonzero((sel >= 0.05) & (sel < 0.1))[:, 0]
    col = torch.randint(0, n, (k,), generator=g, device="cuda")
    A[unb, :, col[unb]] = 0.0                       # one column of zeros with a positive cost: unbounded
    c[unb, col[unb]] = _uniform(g, (len(unb),), 0.5, 1.0)
    ax = torch.einsum("kij,kj->ki", A, x0)
    b = torch.empty((k, m), device="cuda", dtype=torch.float64)
    b[:, :half] = ax[:, :half] + _uniform(g, (k, half), 0.0, 1.0)
    b[:, half:] = _uniform(g, (k, m - half), 0.0, 0.5) - ax[:, half:]
    A[:, half:] *= -1.0
    a = _uniform(g, (len(inf), n), 0.1, 1.0)        # the last two rows contradict each other: infeasible
    beta = (a * x0[inf]).sum(1) + _uniform(g, (len(inf),), 0.0, 1.0)
    A[inf, m - 2], b[inf, m - 2] = a, beta
    A[inf, m - 1], b[inf, m - 1] = -a, -(beta + 1.0)
    return A, b, c


def _mixed_sizes(case):
    r = np.random.default_rng([case["count"], case["lo"], case["hi"]])     # the sizes are the case's, the values the seed's
    return (r.integers(case["lo"], case["hi"] + 1, size=case["count"]),
            r.integers(case["lo"], case["hi"] + 1, size=case["count"]))


def _mixed(case, seed):
    m, n = _mixed_sizes(case)
    g, dt = _gen(seed), DTYPES[case["dtype"]]
    A = _uniform(g, (int((m * n).sum()),), 0.1, 1.0, dt)
    b, c = _uniform(g, (int(m.sum()),), 1.0, 10.0, dt), _uniform(g, (int(n.sum()),), 0.0, 1.0, dt)
    go = torch.randn(case["count"], generator=g, device="cuda", dtype=torch.float64)
    gx = torch.randn(int(n.sum()), generator=g, device="cuda", dtype=torch.float64)
    return m, n, A, b, c, go, gx


def _shared(case, seed):
    g, dt = _gen(seed), DTYPES[case["dtype"]]
    k, m, n = case["count"], case["m"], case["n"]
    A, b = _uniform(g, (m, n), 0.1, 1.0, dt), _uniform(g, (m,), 1.0, 10.0, dt)
    if not case["sweep"]:
        return A, b, _uniform(g, (k, n), 0.0, 1.0, dt)
    c0, d = _uniform(g, (n,), 0.0, 1.0), torch.randn(n, generator=g, device="cuda", dtype=torch.float64)
    steps = 1e-4 * torch.arange(k, device="cuda", dtype=torch.float64)
    return A, b, (c0[None] + steps[:, None] * d[None]).to(dt)


def _bounded(case, seed):
    A, b, c = _type1(case, seed)
    g = _gen(seed + 1_000_003)
    lo = -_uniform(g, c.shape, 0.0, 1.0)
    return A, b, c, lo, lo + _uniform(g, c.shape, 0.5, 2.0)


def _box(case, seed):
    g, dt = _gen(seed), DTYPES[case["dtype"]]
    k, n = case["count"], case["n"]
    shape = (n,) if case["one_box"] else (k, n)
    c = torch.randn((k, n), generator=g, device="cuda", dtype=dt)
    return c, _uniform(g, shape, -10.0, 0.0, dt), _uniform(g, shape, 0.0, 10.0, dt)


def prepare(case, seed):
    kind, s = case["kind"], _solver_()
    if kind in ("dense", "twophase"):
        A, b, c = (_type1 if kind == "dense" else _type2)(case, seed)
        return dict(case=case, solver=s, batch=LPBatch.from_dense(A, b, c))
    if kind == "grad":
        m, n, A, b, c, go, gx = _mixed(case, seed)
        to = lambda v: torch.as_tensor(v, dtype=torch.int32, device="cuda")  # noqa: E731
        return dict(case=case, solver=s, m=to(m), n=to(n), A=A.requires_grad_(), b=b.requires_grad_(),
                    c=c.requires_grad_(), go=go, gx=gx)
    if kind == "shared":
        A, b, C = _shared(case, seed)
        return dict(case=case, solver=s, A=A, b=b, C=C)
    if kind == "bounded":
        A, b, c, lo, up = _bounded(case, seed)
        return dict(case=case, solver=s, batch=LPBatch.from_dense(A, b, c), lo=lo.view(-1), up=up.view(-1))
    if kind == "box":
        c, lo, up = _box(case, seed)
        return dict(case=case, solver=s, c=c, lo=lo, up=up)
    d = LPBatch.from_dense(*_type1(case, seed))     # host: the batch and its results in page-locked memory
    host = LPBatch(*(t.cpu().pin_memory() for t in (d.m, d.n, d.a_off, d.b_off, d.c_off, d.A, d.b, d.c)),
                   d.max_m, d.max_n, d.min_m, d.min_n)
    return dict(case=case, solver=s, batch=host, out=s.alloc_host_result(host))


# ---- one pass ---------------------------------------------------------------

def run(state):
    case, s = state["case"], state["solver"]
    kind = case["kind"]
    if kind in ("dense", "twophase"):
        r = s.solve(state["batch"], prec=case["prec"], pivot_rule=case["rule"])
        if case["rule"] == "steepest":     # its weights are summed in no fixed order: the path may differ between runs
            return dict(status=r.status, obj=r.obj, x=r.x, y=r.y)
        return dict(status=r.status, iters=r.iters, obj=r.obj, x=r.x, y=r.y, basis=r.basis)
    if kind == "grad":
        A, b, c = state["A"], state["b"], state["c"]
        obj, x, y, status = solve(A, b, c, state["m"], state["n"], solver=s)
        loss = (obj * state["go"]).sum() + (x * state["gx"]).sum()
        gA, gb, gc = torch.autograd.grad(loss, (A, b, c))
        return dict(status=status, obj=obj, x=x, y=y, gA=gA, gb=gb, gc=gc)
    if kind == "shared":                   # each objective starts from whichever basis its block held: no fixed path
        r = s.solve_shared(state["A"], state["b"], state["C"], prec=case["prec"])
        return dict(status=r.status, obj=r.obj, x=r.x, y=r.y)
    if kind == "bounded":
        r = s.solve_bounded(state["batch"], state["lo"], state["up"], prec=case["prec"])
        return dict(status=r.status, iters=r.iters, obj=r.obj, x=r.x, y=r.y)
    if kind == "box":
        obj, x = s.hyperbox(state["c"], state["lo"], state["up"], want_x=True)
        return dict(obj=obj, x=x)
    r = s.solve_host(state["batch"], prec=case["prec"], out=state["out"])
    return dict(status=r.status, iters=r.iters, obj=r.obj, x=r.x, y=r.y, basis=r.basis)


# ---- what a pass cannot do without ------------------------------------------

def _lp_work(count, mn, m, n, es, pivots):
    """Inputs read and results written once; 4 m n flops of the two products A x and A^T y that
    check a solution, and per pivot a column and a row of a tableau after the pivots before it
    (or the whole tableau, where that is less)."""
    size = mn / max(1.0, float(count))
    mm, nn = m / max(1, count), n / max(1, count)
    per = min(pivots * (mm + nn), 2.0 * size)
    return dict(bytes=(mn + m + n) * es + (m + n + count) * 8 + 4 * (m + 2 * count), flops=4.0 * mn + count * pivots * per)


def work(case):
    kind = case["kind"]
    es = 4 if case.get("dtype") == "f32" else 8
    if kind == "box":
        k, n = case["count"], case["n"]
        return dict(bytes=(k * n * 2 + (2 * n if case["one_box"] else 2 * k * n) + k) * es, flops=2 * k * n)
    if kind == "grad":
        k, mean = case["count"], (case["lo"] + case["hi"]) / 2.0
        mn = k * mean * mean
        w = _lp_work(k, mn, k * mean, k * mean, es, 0.13 * mean)
        # backward: reads basis, x, y and the upstream gradients, writes dense gradients
        return dict(bytes=w["bytes"] + (mn + 2 * k * mean) * es + 8 * (4 * k * mean + k), flops=w["flops"] + 2 * mn)
    k, m, n = case["count"], case["m"], case["n"]
    pivots = 7.0 * min(m, n) if kind == "twophase" else 0.13 * min(m, n) + 1
    if kind == "shared":
        w = _lp_work(k, k * m * n, k * m, k * n, es, pivots)
        return dict(bytes=(m * n + m + k * n) * es + (k * (m + n + 1)) * 8 + 4 * k, flops=w["flops"])
    w = _lp_work(k, k * m * n, k * m, k * n, es, pivots)
    return dict(bytes=w["bytes"] + (2 * k * n * 8 if kind == "bounded" else 0), flops=w["flops"])


# ---- the results in 64 bits, by plain torch ---------------------------------

def _simplex64(A, b, c):
    """Status (0 optimal, 1 infeasible, 2 unbounded) and optimal basis (a variable per row: j < n
    structural, n + i the slack of row i) of every LP max c x, A x <= b, x >= 0: a dense FP64
    exchange tableau with one auxiliary variable for infeasible starts, batched."""
    K, m, n = A.shape
    dev, X0, eps = A.device, n + m, 1e-9
    status = torch.zeros(K, dtype=torch.int32, device=dev)
    out = torch.zeros((K, m), dtype=torch.int64, device=dev)
    T = torch.zeros((K, m + 2, n + 2), dtype=torch.float64, device=dev)     # rows: constraints, objective, auxiliary
    T[:, :m, :n], T[:, :m, n], T[:, :m, n + 1] = A, -1.0, b
    T[:, m, :n], T[:, m + 1, n] = -c, 1.0
    bas = (n + torch.arange(m, device=dev)).expand(K, m).clone()
    nb = torch.cat([torch.arange(n, device=dev), torch.tensor([X0], device=dev)]).expand(K, n + 1).clone()
    ids, scale = torch.arange(K, device=dev), 1.0 + b.abs().amax(1)

    def pivot(l, e, act):
        at = torch.arange(len(T), device=dev)
        row, col = T[at, l].clone(), T[at, :, e].clone()
        p = torch.where(act, row[at, e], torch.ones_like(row[:, 0]))
        f = torch.where(act[:, None], col / p[:, None], torch.zeros_like(col))
        f[at, l] = 0.0
        torch.baddbmm(T, f.unsqueeze(2), row.unsqueeze(1), alpha=-1.0, out=T)
        T[at, :, e] = torch.where(act[:, None], -f, col)
        new = row / p[:, None]
        new[at, e] = 1.0 / p
        T[at, l] = torch.where(act[:, None], new, row)
        v, w = bas[at, l].clone(), nb[at, e].clone()
        bas[at, l], nb[at, e] = torch.where(act, w, v), torch.where(act, v, w)

    low, first = b.min(1)
    phase = torch.where(low < 0, 1, 2)
    pivot(first, torch.full_like(first, n), phase == 1)
    live = torch.ones(K, dtype=torch.bool, device=dev)
    for _ in range(60 * (m + n)):
        at = torch.arange(len(T), device=dev)
        r = torch.where((nb == X0) & (phase == 2)[:, None], 0.0, T[at, torch.where(phase == 1, m + 1, m), :n + 1])
        v, e = r.min(1)
        stop = live & (v >= -eps)
        if bool((stop & (phase == 1)).any()):          # the auxiliary optimum: feasible, or not
            done1 = stop & (phase == 1)
            bad = done1 & (T[:, m + 1, n + 1].abs() > 1e-8 * scale)
            status[ids[bad]] = 1
            live = live & ~bad
            still = (bas == X0) & (done1 & ~bad)[:, None]
            has = still.any(1)
            if bool(has.any()):                         # the auxiliary variable at zero leaves the basis
                l0 = still.to(torch.int8).argmax(1)
                e0 = torch.where(nb == X0, 0.0, T[at, l0, :n + 1].abs()).argmax(1)
                pivot(l0, e0, has)
            phase = torch.where(done1, 2, phase)
        fin = stop & ~(phase == 1) & (v >= -eps)
        fin = fin & (torch.where(nb == X0, 0.0, T[:, m, :n + 1]).amin(1) >= -eps)
        out[ids[fin]] = bas[fin]
        live = live & ~fin
        go = live & ~stop
        col, rhs = T[at, :m, e], T[:, :m, n + 1]
        ratio = torch.where(col > eps, rhs.clamp_min(0) / col.clamp_min(eps), torch.inf)
        ratio = torch.where((bas == X0) & (ratio <= ratio.amin(1, keepdim=True) + 1e-12), -1.0, ratio)
        q, l = ratio.min(1)
        unb = go & torch.isinf(q)
        status[ids[unb]] = 2
        live = live & ~unb
        pivot(l, e, go & ~unb)
        alive = int(live.sum())
        if alive == 0:
            return status, out
        if alive < 0.7 * len(T):
            T, bas, nb, ids, phase, scale = T[live], bas[live], nb[live], ids[live], phase[live], scale[live]
            live = torch.ones(alive, dtype=torch.bool, device=dev)
    raise RuntimeError("no optimum found")


def _vertex64(A, b, c, status, basis, gx=None):
    """obj, x, y of the basis by FP64 linear solves; with gx also v = B^-T gx_B."""
    K, m, n = A.shape
    step = max(1, 400_000_000 // (m * m * 8))
    obj = torch.empty(K, dtype=torch.float64, device=A.device)
    x, y, w = (torch.zeros(s, dtype=torch.float64, device=A.device) for s in ((K, n), (K, m), (K, m)))
    eye = torch.eye(m, dtype=torch.float64, device=A.device)
    for k in range(0, K, step):
        s = slice(k, k + step)
        ok = (status[s] == 0)[:, None]
        var = basis[s]
        a = torch.gather(A[s], 2, var.clamp_max(n - 1)[:, None, :].expand(-1, m, -1))
        u = eye[(var - n).clamp_min(0)].transpose(1, 2)
        B = torch.where(ok[:, :, None], torch.where((var < n)[:, None, :], a, u), eye)
        put = lambda v: torch.where(var < n, torch.gather(v, 1, var.clamp_max(n - 1)), 0.0)  # noqa: E731
        xb = torch.linalg.solve(B, b[s].unsqueeze(2))[:, :, 0]
        rhs = torch.stack([put(c[s])] + ([put(gx[s])] if gx is not None else []), 2)
        dual = torch.linalg.solve(B.transpose(1, 2), rhs)
        full = torch.zeros((len(var), n + m), dtype=torch.float64, device=A.device).scatter_(1, var, xb)
        x[s] = torch.where(ok, full[:, :n], 0.0)
        y[s] = torch.where(ok, dual[:, :, 0], 0.0)
        if gx is not None:
            w[s] = torch.where(ok, dual[:, :, 1], 0.0)
    obj = (c * x).sum(1)
    obj = torch.where(status == 1, -torch.inf, torch.where(status == 2, torch.inf, obj))
    return obj, x, y, w


def exact(case, seed):
    kind = case["kind"]
    if kind == "box":
        c, lo, up = (t.double() for t in _box(case, seed))
        h = torch.where(c < 0, lo, up)
        return dict(obj=(c * h).sum(1), x=h)
    if kind == "grad":
        return _exact_grad(case, seed)
    if kind == "shared":
        A, b, C = (t.double() for t in _shared(case, seed))
        k, m, n = case["count"], case["m"], case["n"]
        parts = []                         # in blocks: every direction gets its own copy of A here
        for s in range(0, k, 20_000):
            Ak, ck = A.expand(len(C[s:s + 20_000]), m, n), C[s:s + 20_000]
            bk = b.expand(len(ck), m)
            status, basis = _simplex64(Ak, bk, ck)
            parts.append(_vertex64(Ak, bk, ck, status, basis)[:3])
        obj, x, y = (torch.cat(p) for p in zip(*parts))
        return dict(status=None, obj=obj, x=x.view(-1), y=y.view(-1))
    if kind == "bounded":
        A, b, c, lo, up = _bounded(case, seed)
        k, m, n = A.shape
        A2 = torch.cat([A, torch.eye(n, dtype=torch.float64, device="cuda").expand(k, n, n)], 1)
        b2 = torch.cat([b - torch.einsum("kij,kj->ki", A, lo), up - lo], 1)
        status, basis = _simplex64(A2, b2, c)
        obj, z, y, _ = _vertex64(A2, b2, c, status, basis)
        ok = (status == 0)[:, None]
        return dict(status=None, iters=None, obj=obj + (c * lo).sum(1), x=torch.where(ok, z + lo, 0.0).view(-1),
                    y=y[:, :m].reshape(-1))
    A, b, c = (t.double() for t in (_type2 if kind == "twophase" else _type1)(case, seed))
    status, basis = _simplex64(A, b, c)
    obj, x, y, _ = _vertex64(A, b, c, status, basis)
    return dict(status=None, iters=None, obj=obj, x=x.view(-1), y=y.view(-1), basis=None)


def _exact_grad(case, seed):
    m, n, A, b, c, go, gx = _mixed(case, seed)
    k, M, N = case["count"], int(m.max()), int(n.max())
    mt, nt = (torch.as_tensor(v, device="cuda")[:, None] for v in (m, n))
    rows, cols = torch.arange(M, device="cuda")[None] < mt, torch.arange(N, device="cuda")[None] < nt
    both = rows[:, :, None] & cols[:, None, :]
    Ad = torch.zeros((k, M, N), dtype=torch.float64, device="cuda").masked_scatter_(both, A.double())
    pad = lambda mask, v, fill: torch.full(mask.shape, fill, dtype=torch.float64, device="cuda").masked_scatter_(  # noqa: E731
        mask, v.double())
    bd, cd, gd = pad(rows, b, 1.0), pad(cols, c, 0.0), pad(cols, gx, 0.0)     # added rows never bind, columns never enter
    status, basis = _simplex64(Ad, bd, cd)
    obj, x, y, v = _vertex64(Ad, bd, cd, status, basis, gd)
    w = go[:, None] * y + v
    gA = -w[:, :, None] * x[:, None, :]
    return dict(status=None, obj=obj, x=x[cols], y=y[rows], gA=gA[both], gb=w[rows], gc=(go[:, None] * x)[cols])
