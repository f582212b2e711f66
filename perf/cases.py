"""The work whose speed counts: solves, mixed-precision solves, batches, gradients and setup.

Every case goes through the package's public entry points (`lp.LP`, `lp.LPBatch`,
`autodiff.unrolled_pdhg`, `autodiff.unrolled_pdhg_batch`) on seeded LPs of the kinds the package is
used for: standard-form LPs (5 nonzeros per column), LPs with mixed rows and bounds and power-law
column lengths, multicommodity flows on a grid, LPs with one dense row and column, box-bounded LPs.
The data are drawn on the GPU; a program that keeps a handle holds it in its state, and one that
sets up a new LP on each call (the gradients, the setup case) holds the data.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2105_12715_gb300 import autodiff, lp, lpgen

DEV = "cuda"
F64 = torch.float64
EQ, GE, LE = lpgen.ROW_EQ, lpgen.ROW_GE, lpgen.ROW_LE
SCHEMES = {"none": lp.LP_RESTART_NONE, "adaptive": lp.LP_RESTART_ADAPTIVE,
           "flexible": lp.LP_RESTART_FLEXIBLE}
TOL = 1e-8
CHECK_EVERY = 64
ON_CHIP = 129e6  # bytes of L2: a larger problem is read from HBM again in every iteration


def _solve(name, form, m, n, iters, omega=1.0, precision="fp64", scheme="adaptive"):
    return {"name": name, "call": "solve", "form": form, "m": m, "n": n, "iters": iters,
            "omega": omega, "precision": precision, "scheme": scheme}


def listed():
    return [
        # the smallest solve: one tiny LP, a few checks; launches and latency only
        _solve("tiny", "standard", 200, 400, 256),
        # a small LP under the flexible scheme (both candidates' gaps at every check)
        _solve("small_flexible", "mixed", 1999, 9973, 1024, scheme="flexible"),
        # an everyday LP with the primal weight its grid search picks
        _solve("medium", "mixed", 5000, 25000, 1024, omega=0.0625),
        # the next size up, FP32-mixed iterations with FP64 refinement
        _solve("medium_fp32", "mixed", 20000, 100000, 1024, omega=0.0625, precision="mixed"),
        # the package's benchmark LP: 10 million nonzeros, larger than L2
        _solve("large", "mixed", 200000, 1000000, 256, omega=0.0625),
        # the same LP in mixed precision
        _solve("large_fp32", "mixed", 200000, 1000000, 256, omega=0.0625, precision="mixed"),
        # a structured network LP: multicommodity flow, 300 x 300 grid, 8 commodities
        _solve("network", "flow", 300, 8, 256, omega=64.0),
        # one dense row and one dense column among short ones
        _solve("dense_lines", "dense", 20000, 200000, 512),
        # many tiny LPs as one batch
        {"name": "tiny_batch", "call": "batch", "count": 512, "m_lo": 200, "m_hi": 200,
         "iters": 512, "precision": "fp64"},
        # a batch of uneven LPs, 50 to 20,000 rows
        {"name": "uneven_batch", "call": "batch", "count": 96, "m_lo": 50, "m_hi": 20000,
         "iters": 256, "precision": "fp64"},
        # forward and backward of the unrolled solve of one box LP (a differentiable layer)
        {"name": "gradient", "call": "gradient", "count": 1, "m": 2000, "n": 5000, "per_col": 10,
         "iters": 512},
        # a new LP from host arrays: setup, a short solve, the solution back on the host
        {"name": "setup", "call": "setup", "form": "mixed", "m": 100000, "n": 500000,
         "iters": 128},
    ]


def _spread(rng, lo, hi):
    """A whole number in [lo, hi], even over the logarithm."""
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    call = rng.choice(["solve"] * 5 + ["batch"] * 2 + ["gradient", "setup"])
    if call == "solve":
        form = rng.choice(["standard", "mixed", "mixed", "flow", "dense"])
        iters = rng.choice([256, 512, 1024])
        if form == "flow":
            m, n = _spread(rng, 10, 300), rng.randint(2, 8)
        elif form == "dense":
            m = _spread(rng, 1000, 20000)
            n = int(m * rng.uniform(2.0, 10.0))
        else:
            m = _spread(rng, 100, 200000)
            n = int(m * rng.uniform(1.5, 5.0))
        if m > 20000 or (form == "flow" and m > 120):
            iters = 256
        return {"call": "solve", "form": form, "m": m, "n": n, "iters": iters,
                "omega": 64.0 if form == "flow" else rng.choice([0.0625, 0.25, 1.0]),
                "precision": rng.choice(["fp64", "fp64", "mixed"]),
                "scheme": rng.choice(["adaptive", "adaptive", "flexible", "none"])}
    if call == "batch":
        if rng.random() < 0.5:
            m = _spread(rng, 60, 1000)
            return {"call": "batch", "count": _spread(rng, 16, 512 if m <= 300 else 128),
                    "m_lo": m, "m_hi": m, "iters": 256,
                    "precision": rng.choice(["fp64", "mixed"])}
        return {"call": "batch", "count": _spread(rng, 8, 96), "m_lo": 50,
                "m_hi": _spread(rng, 2000, 20000), "iters": 256,
                "precision": rng.choice(["fp64", "mixed"])}
    if call == "gradient":
        m = _spread(rng, 100, 4000)
        return {"call": "gradient", "count": rng.choice([1, 1, 1, rng.randint(2, 16)]), "m": m,
                "n": int(m * rng.uniform(1.5, 3.0)), "per_col": rng.randint(3, 12),
                "iters": rng.choice([128, 256, 512])}
    m = _spread(rng, 1000, 100000)
    return {"call": "setup", "form": rng.choice(["standard", "mixed"]), "m": m,
            "n": int(m * rng.uniform(1.5, 5.0)), "iters": 128}


# ------------------------------------------------------------------ data


def _rand(g, size, lo=0.0, hi=1.0):
    return torch.rand(size, generator=g, device=DEV, dtype=F64) * (hi - lo) + lo


def _randn(g, size):
    return torch.randn(size, generator=g, device=DEV, dtype=F64)


def _zeros(size):
    return torch.zeros(size, device=DEV, dtype=F64)


def _sum_by(which, v, size):
    """Sums of v by group, in a fixed order: the same seed gives the same bits."""
    o = torch.argsort(which, stable=True)
    return torch.segment_reduce(v[o], "sum", lengths=torch.bincount(which, minlength=size))


def _mv(A, v):
    """A v over the nonzeros (rows, cols, vals, m, n)."""
    return _sum_by(A[0], A[2] * v[A[1]], A[3])


def _mtv(A, v):
    return _sum_by(A[1], A[2] * v[A[0]], A[4])


def _pattern(g, degree, row0, nrow, m):
    """Distinct uniform rows per column, column by column (repeats are dropped): rows, cols."""
    cols = torch.repeat_interleave(torch.arange(degree.shape[0], device=DEV), degree)
    u = torch.rand(cols.shape[0], generator=g, device=DEV, dtype=F64)
    rows = row0[cols] + torch.minimum((u * nrow[cols]).long(), nrow[cols] - 1)
    key = torch.unique(cols * m + rows)
    return key % m, key // m


def _csr(A):
    rows, cols, vals, m, n = A
    order = torch.argsort(rows * n + cols)
    ptr = torch.zeros(m + 1, dtype=torch.int64, device=DEV)
    ptr[1:] = torch.cumsum(torch.bincount(rows, minlength=m), 0)
    return ptr.int(), cols[order].int(), vals[order].contiguous()


def _data(A, c, b, lb, ub, rt, px=None, py=None, count=1):
    """The LP on the GPU, and which of `count` problems each column and row belongs to."""
    rows, cols, vals, m, n = A
    ptr, idx, val = _csr(A)
    d = lpgen.LPData(m, n, ptr, idx, val, c, b, lb, ub, rt)
    px = torch.zeros(n, dtype=torch.int64, device=DEV) if px is None else px
    py = torch.zeros(m, dtype=torch.int64, device=DEV) if py is None else py
    return {"lp": d, "A": A, "px": px, "py": py, "count": count}


def _planted_standard(g, A, upper):
    """Ax = b, 0 <= x <= upper, with a planted optimum: x* zero on about half of the columns."""
    m, n = A[3], A[4]
    pos = _rand(g, n) < 0.5
    x = torch.where(pos, _rand(g, n), _zeros(n))
    s = torch.where(pos, _zeros(n), _rand(g, n))
    b, c = _mv(A, x), _mtv(A, _randn(g, m)) + s
    return c, b, _zeros(n), torch.full((n,), upper, device=DEV, dtype=F64), torch.zeros(
        m, dtype=torch.int8, device=DEV)


def _standard(g, m, n, per_col=5, upper=math.inf):
    one = torch.ones(n, dtype=torch.int64, device=DEV)
    rows, cols = _pattern(g, one * min(per_col, m), 0 * one, one * m, m)
    A = (rows, cols, _randn(g, rows.shape[0]), m, n)
    return _data(A, *_planted_standard(g, A, upper))


def _power_law(g, n, kmax):
    k = torch.arange(2, kmax + 1, device=DEV, dtype=F64)
    return torch.multinomial(k ** -1.82, n, replacement=True, generator=g) + 2


def _planted_mixed(g, A):
    """70% EQ / 30% GE rows (half of them active), columns 40% [0, inf), 40% [0, U], 20% free."""
    m, n = A[3], A[4]
    kind, sel, u01 = _rand(g, n), _rand(g, n), _rand(g, n)
    half, box, free = kind < 0.4, (kind >= 0.4) & (kind < 0.8), kind >= 0.8
    inf = torch.full((n,), math.inf, device=DEV, dtype=F64)
    ub = torch.where(box, _rand(g, n, 1.0, 10.0), inf)
    lb = torch.where(free, -inf, _zeros(n))
    zero = _zeros(n)
    at_lo = (half & (sel < 0.5)) | (box & (sel < 1 / 3))
    at_hi = box & (sel >= 2 / 3)
    x = torch.where(half, u01, torch.where(box, u01 * torch.where(box, ub, zero), _randn(g, n)))
    x = torch.where(at_lo, zero, torch.where(at_hi, ub, x))
    s = _rand(g, n)
    s = torch.where(at_lo, s, torch.where(at_hi, -s, zero))
    ge, active = _rand(g, m) < 0.3, _rand(g, m) < 0.5
    y = _randn(g, m)
    y = torch.where(ge, torch.where(active, y.abs(), _zeros(m)), y)
    b = _mv(A, x) - torch.where(ge & ~active, _rand(g, m), _zeros(m))
    return _mtv(A, y) + s, b, lb, ub, torch.where(ge, GE, EQ).to(torch.int8)


def _mixed(g, m, n, dense=False):
    one = torch.ones(n, dtype=torch.int64, device=DEV)
    rows, cols = _pattern(g, _power_law(g, n, min(200, m)), 0 * one, one * m, m)
    if dense:  # row m over all columns, column n over all rows
        rows = torch.cat([rows, torch.full((n,), m, device=DEV), torch.arange(m + 1, device=DEV)])
        cols = torch.cat([cols, torch.arange(n, device=DEV), torch.full((m + 1,), n, device=DEV)])
        m, n = m + 1, n + 1
    A = (rows, cols, _randn(g, rows.shape[0]), m, n)
    return _data(A, *_planted_mixed(g, A))


def _flow(g, side, commodities):
    """Multicommodity min-cost flow on a side x side grid, arcs both ways between neighbours."""
    V = side * side
    at = torch.arange(V, device=DEV).reshape(side, side)
    tail = torch.cat([at[:, :-1].ravel(), at[:, 1:].ravel(), at[:-1].ravel(), at[1:].ravel()])
    head = torch.cat([at[:, 1:].ravel(), at[:, :-1].ravel(), at[1:].ravel(), at[:-1].ravel()])
    arcs = tail.shape[0]
    k = torch.arange(commodities, device=DEV)[:, None]
    col = (k * arcs + torch.arange(arcs, device=DEV)).ravel()
    rows = torch.cat([(k * V + tail).ravel(), (k * V + head).ravel(),
                      (commodities * V + torch.arange(arcs, device=DEV)).repeat(commodities)])
    one = torch.ones(col.shape[0], device=DEV, dtype=F64)
    m, n = commodities * V + arcs, commodities * arcs
    A = (rows, torch.cat([col, col, col]), torch.cat([one, -one, one]), m, n)
    b = _zeros(m)
    for i in range(commodities):
        s, t = torch.randperm(V, generator=g, device=DEV)[:2]
        d = _rand(g, 1, 1.0, 20.0)[0]
        b[i * V + s], b[i * V + t] = d, -d
    b[commodities * V:] = _rand(g, arcs, 5.0, 50.0)
    rt = torch.full((m,), EQ, dtype=torch.int8, device=DEV)
    rt[commodities * V:] = LE
    c = _rand(g, arcs, 1.0, 10.0).repeat(commodities)
    return _data(A, c, b, _zeros(n), torch.full((n,), math.inf, device=DEV, dtype=F64), rt)


def _batch(g, ms, ns, lo, hi, upper):
    """Standard-form LPs of ms[k] rows and ns[k] columns, lo..hi nonzeros per column, as one
    block-diagonal LP."""
    ms, ns = torch.tensor(ms, device=DEV), torch.tensor(ns, device=DEV)
    count, m, n = ms.shape[0], int(ms.sum()), int(ns.sum())
    which = torch.arange(count, device=DEV)
    px, py = torch.repeat_interleave(which, ns), torch.repeat_interleave(which, ms)
    row0 = torch.cumsum(ms, 0) - ms
    degree = torch.minimum(torch.randint(lo, hi + 1, (n,), generator=g, device=DEV), ms[px])
    rows, cols = _pattern(g, degree, row0[px], ms[px], m)
    A = (rows, cols, _randn(g, rows.shape[0]), m, n)
    return _data(A, *_planted_standard(g, A, upper), px, py, count)


def _problems(P):
    """The batch as a list of LPs on the host, as LPBatch takes them."""
    d, out = P["lp"], []
    ptr, idx, val, c, b, lb, ub, rt = (np.asarray(t.cpu()) for t in (
        d.row_ptr, d.col_idx, d.val, d.c, d.b, d.lb, d.ub, d.row_type))
    r1 = np.cumsum(np.asarray(torch.bincount(P["py"], minlength=P["count"]).cpu()))
    c1 = np.cumsum(np.asarray(torch.bincount(P["px"], minlength=P["count"]).cpu()))
    r0 = c0 = 0
    for k in range(P["count"]):
        e0, e1 = ptr[r0], ptr[r1[k]]
        out.append(lpgen.LPData(int(r1[k] - r0), int(c1[k] - c0), ptr[r0:r1[k] + 1] - e0,
                                idx[e0:e1] - c0, val[e0:e1], c[c0:c1[k]], b[r0:r1[k]],
                                lb[c0:c1[k]], ub[c0:c1[k]], rt[r0:r1[k]]))
        r0, c0 = int(r1[k]), int(c1[k])
    return out


def _make(case, seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    if case["call"] == "batch":
        u = np.random.default_rng(12345).uniform(size=case["count"])  # sizes belong to the case
        ms = np.round(case["m_lo"] * (case["m_hi"] / case["m_lo"]) ** u).astype(int).tolist()
        even = case["m_lo"] == case["m_hi"]
        return _batch(g, ms, [2 * m for m in ms], 5 if even else 3, 5 if even else 12, math.inf)
    if case["call"] == "gradient":
        k = case["count"]
        if k == 1:
            return _standard(g, case["m"], case["n"], case["per_col"], 1.0)
        return _batch(g, [case["m"]] * k, [case["n"]] * k, case["per_col"], case["per_col"], 1.0)
    form, m, n = case["form"], case["m"], case["n"]
    if form == "flow":
        return _flow(g, m, n)
    return _standard(g, m, n) if form == "standard" else _mixed(g, m, n, form == "dense")


def _options(case):
    prec = lp.LP_PRECISION_MIXED if case.get("precision") == "mixed" else lp.LP_PRECISION_FP64
    return {"precision": prec, "max_iter": case["iters"], "omega": case.get("omega", 1.0),
            "restart_scheme": SCHEMES[case.get("scheme", "adaptive")],
            "check_every": CHECK_EVERY}


# one check period for every problem, so that a batch repeats its own results
TUNING = {"max_k_shift": 0}


def prepare(case, seed):
    P = _make(case, seed)
    d, s = P["lp"], {"case": case}
    if case["call"] == "solve":
        s["solver"] = lp.LP(d, **_options(case))
    elif case["call"] == "batch":
        s["solver"] = lp.LPBatch(_problems(P), tuning=dict(TUNING), **_options(case))
    elif case["call"] == "gradient":
        s["data"] = d if P["count"] == 1 else _problems(P)
        s["c"], s["b"] = d.c.clone().requires_grad_(), d.b.clone().requires_grad_()
        s["wx"], s["wy"] = _loss_weights(P, seed)
    else:
        names = ("row_ptr", "col_idx", "val", "c", "b", "lb", "ub", "row_type")
        host = {k: getattr(d, k).cpu().pin_memory() for k in names}
        s["data"] = lpgen.LPData(d.m, d.n, **host)
        s["x"] = torch.empty(d.n, dtype=F64).pin_memory()
        s["y"] = torch.empty(d.m, dtype=F64).pin_memory()
    if case["call"] in ("solve", "batch"):
        s["out"] = {k: torch.empty(d.n if k[0] == "x" else d.m, dtype=F64, device=DEV)
                    for k in ("x", "y", "xbar", "ybar", "x0", "y0", "x_sol", "y_sol")}
    return s


def _loss_weights(P, seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed + 1)
    return _randn(g, P["lp"].n), _randn(g, P["lp"].m)


def run(s):
    case = s["case"]
    if case["call"] == "solve":  # from the default start to the tolerance or the iteration limit
        g, o = s["solver"], s["out"]
        g.set_state()
        g.solve(TOL)
        lp.lp_get_solution(g.h, o["x_sol"], o["y_sol"])
        lp.lp_get_state(g.h, o["x"], o["y"], o["xbar"], o["ybar"], o["x0"], o["y0"])
        info = g.info()
        return {**o, "kkt": np.array(info.kkt_avg + info.kkt_cur), "iters": info.iters,
                "restarts": info.restarts}
    if case["call"] == "batch":
        g, o = s["solver"], s["out"]
        g.set_state()
        g.solve(TOL)
        lp.lp_batch_get_solution(g.h, o["x_sol"], o["y_sol"])
        lp.lp_batch_get_state(g.h, o["x"], o["y"], o["xbar"], o["ybar"], o["x0"], o["y0"])
        return dict(o)
    if case["call"] == "gradient":  # a training step through the unrolled solve
        c, b = s["c"], s["b"]
        c.grad = b.grad = None
        if case["count"] == 1:
            x, y = autodiff.unrolled_pdhg(c, b, s["data"], case["iters"], check_every=CHECK_EVERY)
        else:
            x, y = autodiff.unrolled_pdhg_batch(c, b, s["data"], case["iters"],
                                                check_every=CHECK_EVERY, tuning=dict(TUNING))
        ((x * s["wx"]).sum() + (y * s["wy"]).sum()).backward()
        return {"x": x.detach(), "y": y.detach(), "grad_c": c.grad, "grad_b": b.grad}
    with lp.LP(s["data"], **_options(case)) as g:
        g.solve(TOL)
        lp.lp_get_solution(g.h, s["x"], s["y"])
        return {"x": s["x"], "y": s["y"], "iters": g.info().iters}


def work(case):
    """Bytes: a problem that fits in L2 is read once, a larger one once per product and iteration
    (values and indices of A for A^T y and again for A x, each vector of the update read or written
    once).  FLOPs: a multiply and an add per nonzero and product, and the updates."""
    if case["call"] in ("batch", "gradient"):
        count = case["count"]
        if case["call"] == "batch":
            u = np.random.default_rng(12345).uniform(size=count)
            m = int(np.round(case["m_lo"] * (case["m_hi"] / case["m_lo"]) ** u).sum())
            n, per_col = 2 * m, 5.0 if case["m_lo"] == case["m_hi"] else 7.5
        else:
            m, n, per_col = count * case["m"], count * case["n"], float(case["per_col"])
        nnz = n * per_col
    elif case["form"] == "flow":
        arcs = 4 * case["m"] * (case["m"] - 1)
        m, n = case["n"] * case["m"] ** 2 + arcs, case["n"] * arcs
        nnz = 3 * n
    else:
        m, n = case["m"], case["n"]
        nnz = n * (5.0 if case["form"] == "standard" else 10.0)
        if case["form"] == "dense":
            nnz += m + n
    value = 4 if case.get("precision") == "mixed" else 8
    once = nnz * (4 + value) + 6 * value * n + 5 * value * m
    iters = case["iters"]
    twice = 2 * nnz * (4 + value) + 8 * value * n + 6 * value * m
    sweeps = 1 if case["call"] != "gradient" else 3  # forward, recomputed forward, adjoint
    total = twice * iters * sweeps if once > ON_CHIP else once + 8 * 8 * (m + n)
    return {"bytes": total, "flops": iters * sweeps * (4.0 * nnz + 10.0 * n + 8.0 * m)}


# ------------------------------------------------- the same in plain torch


class _Product(torch.autograd.Function):
    """A v by sparse CSR, with A^T for the backward pass."""

    @staticmethod
    def forward(ctx, v, A, AT):
        ctx.AT = AT
        return A @ v

    @staticmethod
    def backward(ctx, g):
        return ctx.AT @ g, None, None


def _sparse(A):
    rows, cols, vals, m, n = A
    fwd = torch.sparse_coo_tensor(torch.stack([rows, cols]), vals, (m, n)).coalesce()
    return fwd.to_sparse_csr(), fwd.t().coalesce().to_sparse_csr()


def _seg(v, which, count):
    return _zeros(count).index_add_(0, which, v)


def _sigma_max(P, A, AT, steps=96):
    """sigma_max of each problem's block: the Lanczos process on A^T A."""
    px, count = P["px"], P["count"]
    g = torch.Generator(device=DEV)
    g.manual_seed(1)
    v, prev, al, be = _rand(g, px.shape[0], 0.5, 1.5), 0.0, [], []
    v = v / _seg(v * v, px, count).sqrt()[px]
    for _ in range(steps):
        w = AT @ (A @ v)
        al.append(_seg(v * w, px, count))
        w = w - al[-1][px] * v - (be[-1][px] * prev if be else 0.0)
        be.append(_seg(w * w, px, count).sqrt())
        prev, v = v, w / be[-1].clamp_min(1e-300)[px]
    T = torch.diag_embed(torch.stack(al, 1)) + torch.diag_embed(torch.stack(be[:-1], 1), 1)
    T = (T + torch.diag_embed(torch.stack(be[:-1], 1), -1)).cpu()
    return torch.linalg.eigvalsh(T)[:, -1].clamp_min(0).sqrt().to(DEV)


def _gap(P, om, lam, gy, x, y, x0, y0):
    """Normalized duality gap of each problem at (x, y), radius its distance to (x0, y0)."""
    d, px, py, count = P["lp"], P["px"], P["py"], P["count"]
    inf, sw = math.inf, math.sqrt(om)
    dx = torch.where(lam > 0, x - d.lb, d.ub - x).clamp_min(0)
    dy = torch.where((gy > 0) & (d.row_type == GE), y.clamp_min(0), torch.where(
        (gy < 0) & (d.row_type == LE), (-y).clamp_min(0), torch.full_like(y, inf)))
    dist, grad = torch.cat([dx * sw, dy / sw]), torch.cat([lam.abs() / sw, gy.abs() * sw])
    which = torch.cat([px, py])
    r2 = om * _seg((x - x0) ** 2, px, count) + _seg((y - y0) ** 2, py, count) / om
    keep = grad > 0
    dist, grad, which = dist[keep], grad[keep], which[keep]
    free = _seg(torch.where(dist.isinf(), grad * grad, 0 * grad), which, count)
    fin = dist.isfinite()
    dist, grad, which = dist[fin], grad[fin], which[fin]
    at = dist / grad
    o = torch.argsort(at)
    o = o[torch.argsort(which[o], stable=True)]
    dist, grad, which, at = dist[o], grad[o], which[o], at[o]

    def cum(v):
        c = torch.cat([_zeros(1), torch.cumsum(v, 0)])
        end = torch.cumsum(torch.bincount(which, minlength=count), 0)
        first = torch.cat([0 * end[:1], end[:-1]])
        return c[1:] - c[first][which], c[end] - c[first]

    d2, g2 = cum(dist * dist)[0], cum(grad * grad)
    f = d2 + at * at * (g2[1][which] - g2[0] + free[which])
    inside = f <= r2[which]
    lo, e_lo = _seg(dist ** 2 * inside, which, count), _seg(dist * grad * inside, which, count)
    hi = _seg(grad ** 2 * ~inside, which, count) + free
    lam_star = torch.where(hi > 0, ((r2 - lo).clamp_min(0) / hi.clamp_min(1e-300)).sqrt(), 0 * hi)
    return torch.where(r2 > 0, (e_lo + lam_star * hi) / r2.clamp_min(1e-300).sqrt(), 0 * r2)


def _reference(P, case, c=None, b=None):
    """Restarted PDHG (Algorithm 1) of every problem in 64 bits."""
    d, px, py, count = P["lp"], P["px"], P["py"], P["count"]
    c, b = d.c if c is None else c, d.b if b is None else b
    A, AT = _sparse(P["A"])
    om, scheme = case.get("omega", 1.0), case.get("scheme", "adaptive")
    eta = 0.9 / _sigma_max(P, A, AT)
    tx, sy = (eta / om)[px], (eta * om)[py]
    tol = 0.0 if case["call"] == "gradient" else TOL
    lo_y = torch.where(d.row_type == GE, 0.0, -math.inf).to(F64)
    hi_y = torch.where(d.row_type == LE, 0.0, math.inf).to(F64)

    def project(v, lo, hi):
        return torch.where((v > lo) & (v < hi), v, torch.minimum(torch.maximum(v, lo), hi).detach())

    x = project(_zeros(d.n), d.lb, d.ub)
    y = _zeros(d.m)
    xb, yb, x0, y0 = x, y, x, y
    nb, nc = _seg(b.detach() ** 2, py, count).sqrt(), _seg(c.detach() ** 2, px, count).sqrt()
    t = torch.zeros(count, dtype=torch.int64, device=DEV)
    restarts, iters = t.clone(), t.clone()
    stored, run_ = _zeros(count), torch.ones(count, dtype=torch.bool, device=DEV)
    cur = torch.zeros(count, dtype=torch.bool, device=DEV)
    kkt = None
    grad = c.requires_grad or b.requires_grad
    for _ in range(case["iters"] // CHECK_EVERY):
        for k in range(CHECK_EVERY):
            w = run_.to(F64) / (t + k + 1).to(F64)
            xn = project(x - tx * (c - _Product.apply(y, AT, A)), d.lb, d.ub)
            yn = project(y + sy * (b - _Product.apply(2 * xn - x, A, AT)), lo_y, hi_y)
            if not grad:  # a problem that has stopped keeps its state
                xn, yn = torch.where(run_[px], xn, x), torch.where(run_[py], yn, y)
            x, y = xn, yn
            xb, yb = xb + w[px] * (x - xb), yb + w[py] * (y - yb)
        with torch.no_grad():
            iters = iters + CHECK_EVERY * run_
            now, gaps = [], []
            for u, v in ((xb, yb), (x, y)):
                lam, gy = c - AT @ v, A @ u - b
                ok = ((lam > 0) & d.lb.isfinite()) | ((lam < 0) & d.ub.isfinite())
                side = torch.where(lam > 0, d.lb, d.ub)
                rp = torch.where(((d.row_type == GE) & (gy > 0)) | ((d.row_type == LE) & (gy < 0)),
                                 0 * gy, gy)
                rp = _seg(rp ** 2, py, count).sqrt()
                rd = _seg(torch.where(ok, 0 * lam, lam) ** 2, px, count).sqrt()
                p = _seg(c * u, px, count)
                dual = _seg(b * v, py, count) + _seg(torch.where(ok, side * lam, 0 * lam), px, count)
                rel = torch.maximum(rp / (1 + nb), rd / (1 + nc))
                rel = torch.maximum(rel, (p - dual).abs() / (1 + p.abs() + dual.abs()))
                now.append(torch.stack([rp, rd, p, dual, rel]))
                gaps.append(_gap(P, om, lam, gy, u, v, x0, y0) if scheme != "none" else None)
            now = torch.cat(now)
            kkt = now if kkt is None else torch.where(run_, now, kkt)
            cur = torch.where(run_, kkt[4] > torch.where(kkt[9] <= tol, tol, kkt[9]), cur)
            go = run_ & ~((kkt[4] <= tol) | (kkt[9] <= tol))
            use = torch.zeros_like(go)
            rho = gaps[0]
            if scheme == "flexible":
                use = go & (gaps[1] < gaps[0])
                rho = torch.where(use, gaps[1], gaps[0])
            t = torch.where(go, t + CHECK_EVERY, t)
            rs = torch.zeros_like(go)
            if scheme != "none":
                rs = go & torch.where(restarts == 0, t >= CHECK_EVERY, rho <= math.exp(-1) * stored)
                stored = torch.where(rs, rho, stored)
            restarts, t, run_ = restarts + rs, torch.where(rs, 0 * t, t), go
        xb, yb = torch.where(use[px], x, xb), torch.where(use[py], y, yb)
        x, y = torch.where(rs[px], xb, x), torch.where(rs[py], yb, y)
        x0, y0 = torch.where(rs[px], xb, x0).detach(), torch.where(rs[py], yb, y0).detach()
        if not grad and not bool(run_.any()):
            break
    return {"x": x, "y": y, "xbar": xb, "ybar": yb, "x0": x0, "y0": y0, "kkt": kkt, "cur": cur,
            "iters": iters, "restarts": restarts}


def exact(case, seed):
    P = _make(case, seed)
    if case["call"] == "gradient":
        d = P["lp"]
        c, b = d.c.clone().requires_grad_(), d.b.clone().requires_grad_()
        r = _reference(P, case, c, b)
        wx, wy = _loss_weights(P, seed)
        ((r["xbar"] * wx).sum() + (r["ybar"] * wy).sum()).backward()
        return {"x": r["xbar"].detach(), "y": r["ybar"].detach(), "grad_c": c.grad,
                "grad_b": b.grad}
    r = _reference(P, case)
    sol = {"x_sol": torch.where(r["cur"][P["px"]], r["x"], r["xbar"]),
           "y_sol": torch.where(r["cur"][P["py"]], r["y"], r["ybar"])}
    if case["call"] == "setup":
        return {"x": sol["x_sol"], "y": sol["y_sol"], "iters": int(r["iters"][0])}
    out = {k: r[k] for k in ("x", "y", "xbar", "ybar", "x0", "y0")}
    out.update(sol)
    if case["call"] == "solve":
        out["kkt"] = np.array(r["kkt"][:, 0].cpu())
        out["iters"], out["restarts"] = int(r["iters"][0]), int(r["restarts"][0])
    return out
