"""The work that is timed: one IPM iteration's linear algebra (or its solves
alone) on the LP families of this repository, through the package's public
entry points.

A case names an LP family with its sizes, the options of the handle and the
entry point.  What a program keeps over an IPM run is kept here too: the
constraint matrix and the analysed handle belong to the case (one handle per
pattern, as in an IPM, where every iteration brings a new Theta and new
right-hand sides), and the seed makes Theta and the right-hand sides.

Families (sizes as in the repository's workloads and tests):
  random      m x n, a fixed number of distinct uniform rows per column, N(0,1)
  grid        multicommodity flow on a side x side 4-neighbour grid, entries +-1
  angular     independent sparse blocks plus dense linking rows
  batch       independent random LPs of log-uniform size, factorised as one forest
  staircase   periods of sparse blocks coupled by identity links

Modes:
  direct      factorise, then a predictor and a corrector solve, device buffers
  solve       one more corrector solve with a factorisation that is there
  graph       the iteration captured once, new inputs copied in, one replay
  host        the iteration from host arrays, results back in host arrays
"""
from __future__ import annotations

from types import SimpleNamespace

import numpy as np
import torch

import paper_2508_04370_gb300 as ipm

RHO = DELTA = 1e-8
NSOLVES = 2  # predictor and one corrector


def listed():
    return [
        # a toy model: every launch and synchronisation shows
        dict(name="random_60x150", family="random", m=60, n=150, per_col=5, decades=4, mode="direct",
             ordering="amd", precision="fp64"),
        # the plain method's LP, late in a run (Theta over 1e-8..1e8)
        dict(name="random_300x800", family="random", m=300, n=800, per_col=6, decades=8, mode="direct",
             ordering="amd", precision="fp64"),
        # the middle of the batch range on its own: a dense root front
        dict(name="random_1537x3843", family="random", m=1537, n=3843, per_col=5, decades=4, mode="direct",
             ordering="amd", precision="fp64"),
        # an ordinary network LP
        dict(name="grid31_amd", family="grid", side=31, commodities=3, decades=6, mode="direct", ordering="amd",
             precision="fp64"),
        # the network benchmark as an IPM loop runs it: one graph replay an iteration
        dict(name="grid64_graph", family="grid", side=64, commodities=4, decades=8, mode="graph", ordering="nd",
             precision="fp64"),
        # multiple centrality correctors: more solves with the same factor
        dict(name="grid64_solve", family="grid", side=64, commodities=4, decades=8, mode="solve", ordering="nd",
             precision="fp64"),
        # block-angular in the normal-equations form, early in a run
        dict(name="angular_normal", family="angular", blocks=37, bm=60, bn=160, density=0.03, linking=8, decades=3,
             form="normal", mode="direct", ordering="amd", precision="fp64"),
        # block-angular with many dense linking rows: thousands of thin fronts
        dict(name="angular_thin", family="angular", blocks=40, bm=150, bn=400, density=0.02, linking=300, decades=3,
             mode="direct", ordering="amd", precision="fp64"),
        # a service that factorises many small LPs at once
        dict(name="batch64", family="batch", count=64, m_lo=100, m_hi=2000, decades=4, mode="direct",
             ordering="amd", precision="fp64"),
        # a multi-period model of ten periods, from and to host arrays
        dict(name="staircase10_host", family="staircase", periods=10, pm=2000, pn=5000, links=500, density=0.002,
             decades=4, mode="host", ordering="nd", precision="sliced"),
        # the same in plain FP64 with device buffers
        dict(name="staircase10_fp64", family="staircase", periods=10, pm=2000, pn=5000, links=500, density=0.002,
             decades=4, mode="direct", ordering="nd", precision="fp64"),
        # the multi-period benchmark at its full size, in the middle of a run
        dict(name="staircase50_graph", family="staircase", periods=50, pm=2000, pn=5000, links=500, density=0.002,
             decades=4, mode="graph", ordering="nd", precision="sliced"),
    ]


def draw(rng):
    """One more case: a family, sizes spread over the logarithm of its range
    (odd ones among them), an entry point, an ordering and a Theta range."""

    def between(lo, hi):
        return max(lo, min(hi, int(round(lo * (hi / lo) ** rng.random()))))

    family = rng.choice(["random", "random", "grid", "grid", "angular", "batch", "staircase"])
    case = dict(family=family, decades=rng.choice([2, 3, 4]), mode=rng.choice(["direct", "direct", "graph", "host", "solve"]),
                ordering="amd", precision="fp64")
    if family == "random":
        m = between(40, 3000)
        case.update(m=m, n=m * 5 // 2 + rng.randrange(7), per_col=rng.choice([4, 5, 6]))
    elif family == "grid":
        case.update(side=between(6, 64), commodities=rng.choice([1, 2, 3, 4]), ordering=rng.choice(["amd", "nd"]))
    elif family == "angular":
        linking = between(2, 200)
        case.update(blocks=between(8, 60), bm=between(20, 150), bn=between(160, 400), density=0.02 + 0.01 * rng.random(),
                    linking=linking)
        if linking <= 10:
            case.update(form="normal", decades=2)
    elif family == "batch":
        case.update(count=between(3, 64), m_lo=50, m_hi=between(200, 2000))
    else:
        pm = between(300, 2000)
        precision = rng.choice(["sliced", "sliced", "fp64"])
        case.update(periods=between(2, 20 if precision == "sliced" else 8), pm=pm, pn=pm * 5 // 2, links=pm // 4,
                    density=4.0 / pm, ordering="nd", precision=precision)
    return case


# ------------------------------------------------------------------ LPs

def _lp(m, n, rows, cols, vals):
    """CSC arrays of a matrix given by distinct (row, column) entries."""
    order = np.argsort(cols.astype(np.int64) * m + rows, kind="stable")
    colptr = np.concatenate([[0], np.cumsum(np.bincount(cols, minlength=n))]).astype(np.int64)
    return SimpleNamespace(m=int(m), n=int(n), colptr=colptr, rowidx=np.ascontiguousarray(rows[order], np.int32),
                           vals=np.ascontiguousarray(vals[order], np.float64))


def _cover(rng, m, n, keys):
    """Entry keys (column * m + row) without repeats, with at least one entry in
    every row and column."""
    keys = np.unique(keys)
    empty = np.setdiff1d(np.arange(m), keys % m)
    keys = np.union1d(keys, rng.integers(n, size=empty.size) * m + empty)
    empty = np.setdiff1d(np.arange(n), keys // m)
    return np.union1d(keys, empty * m + rng.integers(m, size=empty.size))


def _random_lp(m, n, per_col, seed):
    rng = np.random.default_rng(seed)
    k = min(per_col, m)
    rows = rng.integers(m, size=(n, k))
    while True:  # distinct rows in a column: draw the columns with repeats again
        s = np.sort(rows, axis=1)
        bad = np.flatnonzero((s[:, 1:] == s[:, :-1]).any(axis=1))
        if not bad.size:
            break
        rows[bad] = rng.integers(m, size=(bad.size, k))
    keys = _cover(rng, m, n, (np.arange(n)[:, None] * m + rows).reshape(-1))
    return _lp(m, n, keys % m, keys // m, rng.standard_normal(keys.size))


def _grid_lp(side, commodities):
    nodes = side * side
    v = np.arange(nodes).reshape(side, side)
    u = np.concatenate([v[:, :-1].reshape(-1), v[:-1, :].reshape(-1)])
    w = np.concatenate([v[:, 1:].reshape(-1), v[1:, :].reshape(-1)])
    e = np.arange(u.size)
    tail, head, edge = np.concatenate([u, w]), np.concatenate([w, u]), np.concatenate([e, e])
    arcs, cons = tail.size, commodities * (nodes - 1)
    rows, cols, vals = [], [], []
    for q in range(commodities):
        j = q * arcs + np.arange(arcs)
        for node, val in ((tail, 1.0), (head, -1.0)):
            on = node > 0  # node 0's conservation row is dropped
            rows.append(q * (nodes - 1) + node[on] - 1)
            cols.append(j[on])
            vals.append(np.full(int(on.sum()), val))
        rows.append(cons + edge)
        cols.append(j)
        vals.append(np.ones(arcs))
    return _lp(cons + u.size, commodities * arcs, np.concatenate(rows), np.concatenate(cols), np.concatenate(vals))


def _sparse_block(rng, bm, bn, density):
    keys = _cover(rng, bm, bn, rng.integers(bm * bn, size=int(round(bm * bn * density))))
    return keys % bm, keys // bm


def _angular_lp(blocks, bm, bn, density, linking, seed):
    rng = np.random.default_rng(seed)
    rows, cols = [], []
    for b in range(blocks):
        r, c = _sparse_block(rng, bm, bn, density)
        rows.append(r + b * bm)
        cols.append(c + b * bn)
    m, n = blocks * bm + linking, blocks * bn
    rows.append(np.tile(np.arange(blocks * bm, m), n))
    cols.append(np.repeat(np.arange(n), linking))
    rows, cols = np.concatenate(rows), np.concatenate(cols)
    return _lp(m, n, rows, cols, rng.standard_normal(rows.size))


def _staircase_lp(periods, pm, pn, links, density, seed):
    rng = np.random.default_rng(seed)
    rows, cols, vals = [], [], []
    for t in range(periods):
        r, c = _sparse_block(rng, pm, pn, density)
        rows.append(r + t * pm)
        cols.append(c + t * pn)
        vals.append(rng.standard_normal(r.size))
        if t + 1 < periods:
            rows.append(np.arange(links) + (t + 1) * pm)
            cols.append(np.arange(links) + t * pn)
            vals.append(np.ones(links))
    return _lp(periods * pm, periods * pn, np.concatenate(rows), np.concatenate(cols), np.concatenate(vals))


def _lps(case):
    """The case's LP (several for a batch); its values belong to the case."""
    f = case["family"]
    if f == "random":
        return [_random_lp(case["m"], case["n"], case["per_col"], 1)]
    if f == "grid":
        return [_grid_lp(case["side"], case["commodities"])]
    if f == "angular":
        return [_angular_lp(case["blocks"], case["bm"], case["bn"], case["density"], case["linking"], 1)]
    if f == "staircase":
        return [_staircase_lp(case["periods"], case["pm"], case["pn"], case["links"], case["density"], 1)]
    rng = np.random.default_rng(1)
    ms = np.exp(rng.uniform(np.log(case["m_lo"]), np.log(case["m_hi"]), size=case["count"])).round().astype(int)
    return [_random_lp(int(m), int(round(2.5 * m)), 5, 2 + i) for i, m in enumerate(ms)]


# -------------------------------------------------------------- handles

_handles = {}  # the latest case's handle


def _handle(case):
    """The analysed handle a program keeps for the case's pattern."""
    key = repr(sorted((k, v) for k, v in case.items() if k != "name"))
    if key in _handles:
        return _handles[key]
    _handles.clear()  # one pattern at a time; a state in use keeps its own alive
    lps = _lps(case)
    options = dict(precision=ipm.IPM_PREC_SLICED if case["precision"] == "sliced" else ipm.IPM_PREC_FP64)
    ordering = ipm.IPM_ORD_ND if case["ordering"] == "nd" else ipm.IPM_ORD_AMD
    if case["family"] == "batch":
        solver = ipm.BatchSolver(lps, ordering=ordering, **options)
    else:
        form = ipm.IPM_FORM_NORMAL if case.get("form") == "normal" else ipm.IPM_FORM_AUGMENTED
        solver = ipm.Solver.from_lp(lps[0], form=form, ordering=ordering, **options)
    h = SimpleNamespace(solver=solver, lps=lps, m=solver.m, n=solver.n, graph=None, factorised=False)
    _handles[key] = h
    return h


def _vectors(h, case, seed):
    """Theta and the right-hand sides of one IPM iteration, on the GPU."""
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    d = float(case["decades"])
    theta = torch.pow(10.0, d * (2.0 * torch.rand(h.n, dtype=torch.float64, device="cuda", generator=g) - 1.0))
    r7 = torch.randn(NSOLVES * h.n, dtype=torch.float64, device="cuda", generator=g)
    r1 = torch.randn(NSOLVES * h.m, dtype=torch.float64, device="cuda", generator=g)
    return theta, r7, r1


def prepare(case, seed):
    h = _handle(case)
    theta, r7, r1 = _vectors(h, case, seed)
    s = SimpleNamespace(h=h, mode=case["mode"], theta=theta, r7=r7, r1=r1)
    if s.mode == "solve" and not h.factorised:
        # the iteration's factorisation is there already; the seed brings right-hand sides
        h.solver.factorise(_vectors(h, case, 0)[0], RHO, DELTA)
        h.factorised = True
    if s.mode == "graph" and h.graph is None:
        h.graph = SimpleNamespace(theta=theta.clone(), r7=r7.clone(), r1=r1.clone(), dx=torch.empty_like(r7),
                                  dy=torch.empty_like(r1))
        b = h.graph
        rc = ipm.ipm_graph_capture(h.solver.ctx, b.theta, RHO, DELTA, b.r7, b.r1, b.dx, b.dy, nsolves=NSOLVES)
        if rc:
            raise RuntimeError(f"ipm_graph_capture failed ({rc})")
    if s.mode == "host":
        s.theta, s.r7, s.r1 = (t.cpu().numpy() for t in (theta, r7, r1))
    return s


def run(s):
    h, solver = s.h, s.h.solver
    if s.mode == "graph":
        b = h.graph
        b.theta.copy_(s.theta)
        b.r7.copy_(s.r7)
        b.r1.copy_(s.r1)
        rc = ipm.ipm_graph_launch(solver.ctx)
        if rc:
            raise RuntimeError(f"ipm_graph_launch failed ({rc})")
        return b.dx.clone(), b.dy.clone()
    if s.mode == "host":
        dx, dy = np.empty_like(s.r7), np.empty_like(s.r1)
        rc = ipm.ipm_iterate_host(solver.ctx, s.theta, RHO, DELTA, s.r7, s.r1, dx, dy, nrhs=NSOLVES)
        if rc < 0:
            raise RuntimeError(f"ipm_iterate_host failed ({rc})")
        return dx, dy
    if s.mode == "solve":
        return solver.solve(s.r7[: h.n], s.r1[: h.m])
    solver.factorise(s.theta, RHO, DELTA)
    out = [solver.solve(s.r7[k * h.n:(k + 1) * h.n], s.r1[k * h.m:(k + 1) * h.m]) for k in range(NSOLVES)]
    return torch.cat([x for x, _ in out]), torch.cat([y for _, y in out])


def work(case):
    """The inputs read once and the results written once, the factorisation's
    flops on this pattern and two per entry of L and sweep.  L itself, once it
    is larger than the 129 MB L2, is written once and read by both sweeps of
    every solve."""
    h = _handle(case)
    info = h.solver.info()
    nsol = 1 if case["mode"] == "solve" else NSOLVES
    factor = case["mode"] != "solve"
    nnz = info["nnz_L"]
    values = (info["nnz_A"] + h.n) * factor + 2 * nsol * (h.n + h.m)
    if 8 * nnz > 129e6:
        values += nnz * (factor + 2 * nsol)
    return {"bytes": 8.0 * values, "flops": info["flops_factor"] * factor + 4.0 * nnz * nsol}


# ---------------------------------------------------------------- exact

def _dense_solve(lp, theta, r7, r1):
    """(dx, dy) of K [dx; dy] = [r7; r1] by dense factorisations in 64 bits,
    refined to the backward error that 64-bit residuals allow; None where it
    does not get there or the matrices are too large."""
    m, n, dev = lp.m, lp.n, theta.device
    col = torch.as_tensor(np.repeat(np.arange(n), np.diff(lp.colptr)), device=dev)
    row = torch.as_tensor(lp.rowidx.astype(np.int64), device=dev)
    val = torch.as_tensor(lp.vals, device=dev)
    h = 1.0 / theta + RHO
    f = torch.cat([r7, r1])

    def apply(hh, vv, dd, x):
        out = torch.cat([hh * x[:n], dd * x[n:]])
        out.index_add_(0, col, vv * x[n + row])
        out.index_add_(0, n + row, vv * x[col])
        return out

    if n + m <= 12000:
        K = torch.zeros(n + m, n + m, dtype=torch.float64, device=dev)
        K[col, n + row] = val
        K[n + row, col] = val
        K.diagonal().copy_(torch.cat([-h, torch.full((m,), DELTA, dtype=torch.float64, device=dev)]))
        lu = torch.linalg.lu_factor(K)

        def inverse(r):
            return torch.linalg.lu_solve(*lu, r[:, None])[:, 0]
    else:
        ptr = torch.as_tensor(lp.colptr, device=dev)
        deg = ptr[1:] - ptr[:-1]
        S = torch.zeros(m, m, dtype=torch.float64, device=dev)
        if float((deg.double() ** 2).sum()) <= 3e7 and m <= 26000:
            # A H^-1 A^T from the entry pairs of each column
            rep = deg[col]
            a = torch.repeat_interleave(torch.arange(val.numel(), device=dev), rep)
            first = torch.cumsum(rep, 0) - rep
            b = ptr[col[a]] + torch.arange(a.numel(), device=dev) - first[a]
            S.view(-1).index_add_(0, row[a] * m + row[b], val[a] * val[b] / h[col[a]])
        elif 2.0 * m * m * n <= 5e12:
            A = torch.zeros(m, n, dtype=torch.float64, device=dev)
            A[row, col] = val
            S = (A / h) @ A.T
        else:
            return None
        S.diagonal().add_(DELTA)
        C, bad = torch.linalg.cholesky_ex(S)
        if int(bad):
            return None
        del S

        def inverse(r):
            t = torch.zeros(m, dtype=torch.float64, device=dev).index_add_(0, row, val * (r[:n] / h)[col]) + r[n:]
            y = torch.cholesky_solve(t[:, None], C)[:, 0]
            return torch.cat([(torch.zeros_like(h).index_add_(0, col, val * y[row]) - r[:n]) / h, y])

    x, best = inverse(f), None
    for _ in range(30):
        r = f - apply(-h, val, DELTA, x)
        w = float((r.abs() / (apply(h, val.abs(), DELTA, x.abs()) + f.abs()).clamp_min(1e-300)).max())
        if best is None or w < best[0]:
            best = (w, x)
        if w > 2.0 * best[0] or w <= 1e-16:
            break
        x = x + inverse(r)
    return (best[1][:n], best[1][n:]) if best[0] <= 1e-14 else None


def exact(case, seed):
    if case["family"] == "staircase" and case["periods"] * case["pm"] > 26000:
        return None
    h = _handle(case)
    theta, r7, r1 = _vectors(h, case, 0 if case["mode"] == "solve" else seed)
    if case["mode"] == "solve":
        _, r7, r1 = _vectors(h, case, seed)
    dx, dy = [], []
    for k in range(1 if case["mode"] == "solve" else NSOLVES):
        no, mo = k * h.n, k * h.m
        to = 0
        for lp in h.lps:
            got = _dense_solve(lp, theta[to:to + lp.n], r7[no:no + lp.n], r1[mo:mo + lp.m])
            if got is None:
                return None
            dx.append(got[0])
            dy.append(got[1])
            no, mo, to = no + lp.n, mo + lp.m, to + lp.n
    dx, dy = torch.cat(dx), torch.cat(dy)
    return (dx.cpu().numpy(), dy.cpu().numpy()) if case["mode"] == "host" else (dx, dy)
