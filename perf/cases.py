"""The workloads whose speed this repository answers for, each through the public entry points of the binding.

A case is a plain dict.  ``call`` says which entry point a pass goes through: ``solve`` (one batched solve on a handle),
``joint`` (several handles' batches together), ``create`` (a handle from host arrays) or ``serve`` (a burst of requests
to a server).  ``rows`` names the sparsity recipe, ``m``, ``n`` and ``lps`` the sizes, ``iters`` the iteration budget.

Most solves run a fixed budget of iterations, as strong branching does: the same work whatever the inputs.  One runs
until every LP meets its tolerance.  All values, bounds and overrides follow the seeded generators of this repository
(coefficients +-U[0.1, 10], row bounds around a generating point), drawn here on the GPU.
"""
from __future__ import annotations

import math
import types

import numpy as np
import torch

from paper_2601_21990_gb300 import lpb

_FIELDS = ("status", "restarts", "iters", "obj", "dual_obj", "rel_primal", "rel_dual", "rel_gap", "safe_bound")
_WHOLE = ("status", "restarts", "iters")


def _case(name, call, rows, m, n, lps, iters, **more):
    return {"name": name, "call": call, "rows": rows, "m": m, "n": n, "lps": lps, "iters": iters, "precision": "mixed",
            "tol": 1e-4, "polish": False, "parts": 1, **more}


def listed():
    return [
        # the smallest matrix of the tests, in the precision of the paper: launches and latency
        _case("small_fp64", "solve", "columns", 200, 400, 16, 512, precision="fp64"),
        # the smallest serving matrix, a ragged number of children: a node's candidates in branch and bound
        _case("serve1k", "solve", "powerlaw", 1000, 2000, 37, 512),
        # one candidate's up and down child on a middle-sized matrix: the narrowest batch
        _case("one_candidate", "solve", "powerlaw", 20000, 50000, 2, 256),
        # the power-law strong-branching batch, a fixed budget
        _case("powerlaw64", "solve", "powerlaw", 20000, 50000, 64, 256),
        # the same batch until every child has its status: a whole call, checks, compactions and restarts among it
        _case("powerlaw64_whole", "solve", "powerlaw", 20000, 50000, 64, 4000, whole=True),
        # the largest serving matrix, a ragged request
        _case("serve200k", "solve", "powerlaw", 200000, 400000, 101, 64),
        # bound tightening: objectives +-e_j, free variables, 1024 LPs
        _case("obbt1024", "solve", "square", 100000, 100000, 1024, 64),
        # the double-float polish: LPs held to 1e-8 leave FP32 at the second check
        _case("polish", "solve", "square", 10000, 10000, 64, 384, tol=1e-8, polish=True),
        # strong branching on the largest matrix: a million rows, dense rows among them
        _case("large128", "solve", "bimodal", 1000000, 2000000, 128, 64),
        # eight small matrices' batches in joint launches
        _case("joint8", "joint", "powerlaw", 1000, 2000, 32, 256, parts=8),
        # a handle from host arrays: transpose, scaling, step size
        _case("create100k", "create", "square", 100000, 100000, 0, 0),
        # a burst of requests to a server that runs them together
        _case("serve_burst", "serve", "square", 5000, 5000, 24, 128, parts=8),
    ]


def draw(rng):
    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    call = rng.choice(["solve"] * 7 + ["whole", "polish", "joint", "create", "serve"])
    rows = rng.choice(["powerlaw", "powerlaw", "square", "columns", "bimodal"])
    if call == "serve":
        m = log(1000, 20000)
        return _case("", call, "square", m, m, log(4, 48), rng.randint(64, 192), parts=rng.randint(2, 12))
    if call == "joint":
        m = log(200, 5000)
        return _case("", call, rng.choice(["powerlaw", "columns"]), m, 2 * m, log(4, 96), rng.randint(64, 320),
                     parts=rng.randint(2, 10))
    if call == "polish":
        m = log(1000, 30000)
        return _case("", "solve", "square", m, m, log(4, 256), rng.randint(192, 512), tol=1e-8, polish=True)
    if call == "whole":
        m = log(2000, 30000)
        return _case("", "solve", "powerlaw", m, int(m * rng.uniform(1.5, 2.5)), log(4, 128), 4000, whole=True)
    m = log(2000 if rows == "bimodal" else 200, 400000)
    n = m if rows == "square" else int(m * rng.uniform(1.5, 2.5))
    if call == "create":
        return _case("", call, rows, m, n, 0, 0, precision=rng.choice(["mixed", "mixed", "fp64"]))
    c = _case("", call, rows, m, n, log(1, 1024), rng.randint(64, 512),
              precision=rng.choice(["mixed", "mixed", "mixed", "fp64"]))
    slow = 8 if c["precision"] == "fp64" else 1
    while c["lps"] * (_nnz(c) + 3 * (m + n)) * c["iters"] * slow > 8e10 or c["lps"] * n > 2e8:
        if c["iters"] > 128:
            c["iters"] //= 2
        else:
            c["lps"] = (c["lps"] + 1) // 2
    return c


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _dense_rows(m):
    return max(1, m // 2000)


def _nnz(case):
    m, n = case["m"], case["n"]
    return {"powerlaw": 12.5 * m, "square": 10 * m, "columns": 5 * n,
            "bimodal": 5.5 * m + _dense_rows(m) * (n // 200)}[case["rows"]]


def _distinct(g, lengths, width):
    """lengths[i] distinct indices in [0, width) for each i, sorted: (owner, index)."""
    own = torch.repeat_interleave(torch.arange(lengths.numel(), device="cuda"), lengths)
    key = torch.sort(own * width + torch.randint(0, width, (own.numel(),), device="cuda", generator=g))[0]
    while True:
        dup = torch.nonzero(key[1:] == key[:-1]).flatten() + 1
        if dup.numel() == 0:
            return own, key - own * width
        key[dup] = own[dup] * width + torch.randint(0, width, (dup.numel(),), device="cuda", generator=g)
        key = torch.sort(key)[0]


def _uniform(g, lo, hi, *size):
    return torch.rand(*size, dtype=torch.float64, device="cuda", generator=g) * (hi - lo) + lo


def _problem(rows, m, n, seed):
    """One LP on the GPU, FP64: its CSR arrays and vectors, and the point that its row bounds lie around."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    if rows == "columns":  # every column has 4 to 6 rows
        length = torch.randint(4, 7, (n,), device="cuda", generator=g)
        j, i = _distinct(g, length, m)
        key = torch.sort(i * n + j)[0]
        i, j = key // n, key % n
    else:
        if rows == "powerlaw":  # lengths P(k) ~ k^-1.839 on [2, 500]
            k = torch.arange(2, 501, device="cuda")
            p = k.double() ** -1.839
            cut = torch.cumsum(p / p.sum(), 0)
            at = torch.searchsorted(cut, _uniform(g, 0.0, 1.0, m)).clamp(max=498)
            length = k[at].clamp(max=n)
        elif rows == "square":
            length = torch.full((m,), 10, device="cuda")
        else:  # "bimodal": 3 to 8 entries, and one row in 2000 with n / 200
            length = torch.randint(3, 9, (m,), device="cuda", generator=g)
            length[torch.randperm(m, device="cuda", generator=g)[:_dense_rows(m)]] = n // 200
        i, j = _distinct(g, length, n)
    sign = torch.where(_uniform(g, 0.0, 1.0, i.numel()) < 0.5, -1.0, 1.0)
    v = _uniform(g, 0.1, 10.0, i.numel()) * sign
    if rows == "square":  # boxes within [-100, 100], one variable in ten free, no cost
        a, b = _uniform(g, -100.0, 100.0, n), _uniform(g, -100.0, 100.0, n)
        lo, hi = torch.minimum(a, b), torch.maximum(a, b)
        x0 = lo + _uniform(g, 0.0, 1.0, n) * (hi - lo)
        free = _uniform(g, 0.0, 1.0, n) < 0.1
        x0 = torch.where(free, 10.0 * torch.randn(n, dtype=torch.float64, device="cuda", generator=g), x0)
        lo[free], hi[free] = -math.inf, math.inf
        c = torch.zeros(n, dtype=torch.float64, device="cuda")
    else:
        x0 = _uniform(g, 0.0, 10.0, n)
        lo, hi = torch.zeros_like(x0), torch.full_like(x0, 10.0)
        c = torch.randn(n, dtype=torch.float64, device="cuda", generator=g)
    ptr = torch.zeros(m + 1, dtype=torch.int64, device="cuda")
    ptr[1:] = torch.cumsum(torch.bincount(i, minlength=m), 0)
    ax = torch.mv(torch.sparse_csr_tensor(ptr, j, v, (m, n)), x0)
    p = types.SimpleNamespace(m=m, n=n, ptr=ptr, row=i, col=j, val=v, c=c, lo=lo, hi=hi, x0=x0, gen=g)
    p.rl, p.ru = ax - _uniform(g, 0.0, 1.0, m), ax + _uniform(g, 0.0, 1.0, m)
    return p


def _overrides(p, rows, lps):
    """Strong-branching children (all up, then all down), or minima then maxima of variables for "square"."""
    half = (lps + 1) // 2
    var = torch.randperm(p.n, device="cuda", generator=p.gen)[:half].repeat(math.ceil(lps / max(half, 1)))[:lps]
    first = torch.arange(lps, device="cuda") < half
    if rows == "square":
        return lpb.specs_array(np.full(lps, 2), var.cpu().numpy(), sign=torch.where(first, 1.0, -1.0).cpu().numpy())
    x = p.x0[var]
    lo = torch.where(first, torch.ceil(x), torch.full_like(x, -math.inf))
    hi = torch.where(first, torch.full_like(x, math.inf), torch.floor(x))
    return lpb.specs_array(np.ones(lps), var.cpu().numpy(), lo.cpu().numpy(), hi.cpu().numpy())


def _host(p):
    """The LP as the host arrays that a handle is made from."""
    h = {"row_ptr": p.ptr, "col_idx": p.col.int(), "vals": p.val, "c": p.c, "row_lo": p.rl, "row_hi": p.ru,
         "var_lo": p.lo, "var_hi": p.hi}
    return types.SimpleNamespace(m=p.m, n=p.n, **{k: v.cpu().numpy() for k, v in h.items()})


def _options(case):
    o = {"precision": lpb.FP64 if case["precision"] == "fp64" else lpb.MIXED}
    if case["polish"]:
        o["polish_stall_checks"] = 1
    return o


def _inputs(case, seed):
    """The case's problems and the override records of its batches: [(problem, [records, ...]), ...]."""
    m, n, lps, parts = case["m"], case["n"], case["lps"], case["parts"]
    if case["call"] == "joint":  # m, 1.25 m, 1.5 m, ...
        ps = [_problem(case["rows"], m + k * m // 4, n + k * n // 4, 64 * seed + k) for k in range(parts)]
        return [(p, [_overrides(p, case["rows"], lps)]) for p in ps]
    p = _problem(case["rows"], m, n, 64 * seed)
    if case["call"] == "serve":  # requests of lps / 2 to 3 lps / 2 LPs
        sizes = [max(1, lps // 2 + k * lps // max(1, parts - 1)) for k in range(parts)]
        return [(p, [_overrides(p, case["rows"], s) for s in sizes])]
    return [(p, [_overrides(p, case["rows"], lps)])] if lps else [(p, [])]


def prepare(case, seed):
    inputs = _inputs(case, seed)
    s = types.SimpleNamespace(case=dict(case), options=_options(case), lps=[_host(p) for p, _ in inputs],
                              specs=[sp for _, sps in inputs for sp in sps], handles=[])
    del inputs
    torch.cuda.empty_cache()
    if case["call"] != "create":
        s.handles = [lpb.Handle(lp, **s.options) for lp in s.lps]
        s.lps = []  # the handle has its own copy
    if case["call"] == "serve":
        s.server = lpb.Server()
        s.matrix = s.server.attach(s.handles[0])
    return s


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------

class _OnDevice:
    """A batch's result block as an array interface; keeps the batch alive as long as the array is."""

    def __init__(self, batch, ptr, shape):
        self.batch = batch
        self.__cuda_array_interface__ = {"shape": shape, "typestr": "<f8", "data": (ptr, False), "version": 3}


def _fields(results):
    r = np.concatenate(results)
    return {f: np.ascontiguousarray(r[f]) for f in _FIELDS}


def _points(batches):
    xs, ys = [], []
    for b in batches:
        x, y = b.device_xy()
        xs.append(torch.as_tensor(_OnDevice(b, x, (b.num_lps, b.n)), device="cuda"))
        ys.append(torch.as_tensor(_OnDevice(b, y, (b.num_lps, b.m)), device="cuda"))
    return {"x": xs, "y": ys}


def run(state):
    case, call = state.case, state.case["call"]
    if call == "create":
        h = lpb.Handle(state.lps[0], **state.options)
        eta, norm, iters = h.info()
        row, col = h.scaling()
        h.close()
        return {"eta": eta, "norm": norm, "iters": iters, "row": row, "col": col}
    if call == "serve":
        srv = state.server
        ids = [srv.submit(state.matrix, sp, tol=case["tol"], max_iter=case["iters"]) for sp in state.specs]
        for r in ids:
            srv.wait(r)
        points = [srv.result(r, state.matrix, q)[1:] for r, sp in zip(ids, state.specs) for q in range(len(sp))]
        out = _fields([srv.results(r) for r in ids])
        for r in ids:
            srv.release(r)
        return {**out, "x": np.stack([x for x, _ in points]), "y": np.stack([y for _, y in points])}
    if call == "joint":
        batches = lpb.Handle.solve_multi(state.handles, state.specs, tol=case["tol"], max_iter=case["iters"])
    else:
        batches = [state.handles[0].solve(state.specs[0], tol=case["tol"], max_iter=case["iters"])]
    return {**_fields([b.results() for b in batches]), **_points(batches)}


def work(case):
    """An iteration takes two products with the matrix (value and index of every entry, both ways) and reads the
    iterate blocks, their anchors and the bounds once and writes the iterates once; a result is one point.  For a
    solve until the tolerance, 1000 iterations are counted."""
    m, n, lps, nnz, parts = case["m"], case["n"], case["lps"], _nnz(case), case["parts"]
    if case["call"] == "create":  # the matrix in, both orders of the scaled matrix out
        return {"bytes": 12.0 * nnz + 8 * m + 24.0 * nnz + 8.0 * 5 * (m + n), "flops": 4.0 * nnz * 100}
    size = 8 if case["precision"] == "fp64" else 4
    iters = 1000 if case.get("whole") else case["iters"]
    grow = 1.0
    if case["call"] == "joint":
        grow = parts * (1 + (parts - 1) / 8)  # the matrices grow by a quarter from one to the next
    elif case["call"] == "serve":
        lps *= parts
    step = 2 * (4 + size) * nnz + size * lps * 3.0 * (m + n) + 2 * size * (m + n)
    if case["polish"]:  # two of the checked intervals in FP32, the others in pairs of FP32 values
        step = (step * 128 + max(0, iters - 128) * (2 * 12 * nnz + 8 * lps * 3.0 * (m + n))) / max(iters, 128)
    return {"bytes": grow * (iters * step + 8.0 * lps * (m + n)), "flops": grow * 4.0 * nnz * lps * iters}


# ---------------------------------------------------------------------------
# the same in 64 bits, by plain tensor operations
# ---------------------------------------------------------------------------

def _scaled(p):
    """Ten Ruiz passes and one Pock-Chambolle pass, then the power iteration: (d_r, d_c, A~, A~^T, norm, products)."""
    m, n, i, j = p.m, p.n, p.row, p.col
    dr, dc = torch.ones(m, dtype=torch.float64, device="cuda"), torch.ones(n, dtype=torch.float64, device="cuda")
    for k in range(11):
        a = (dr[i] * p.val * dc[j]).abs()
        how = "amax" if k < 10 else "sum"
        sr = torch.zeros_like(dr).scatter_reduce(0, i, a, how)
        sc = torch.zeros_like(dc).scatter_reduce(0, j, a, how)
        dr, dc = torch.where(sr > 0, dr / sr.sqrt(), dr), torch.where(sc > 0, dc / sc.sqrt(), dc)
    v = dr[i] * p.val * dc[j]
    order = torch.argsort(j, stable=True)
    tptr = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    tptr[1:] = torch.cumsum(torch.bincount(j, minlength=n), 0)
    A = torch.sparse_csr_tensor(p.ptr, j, v, (m, n))
    At = torch.sparse_csr_tensor(tptr, i[order], v[order], (n, m))
    # the start vector: SplitMix64 of the default power_seed
    z = np.uint64(0x5EED) + (np.arange(n, dtype=np.uint64) + np.uint64(1)) * np.uint64(0x9E3779B97F4A7C15)
    z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
    z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
    z ^= z >> np.uint64(31)
    w = torch.from_numpy(2.0 * ((z >> np.uint64(11)).astype(np.float64) * 2.0 ** -53) - 1.0).cuda()
    prev, norm, k = -1.0, 0.0, 0
    for k in range(1, 5001):
        u = torch.mv(A, w / w.norm())
        norm = float(u.norm())
        w = torch.mv(At, u)
        if prev >= 0 and abs(norm - prev) <= 1e-10 * norm:
            break
        prev = norm
    return dr, dc, A, At, norm, k


def _barrier(v, a, b):
    """Onto the cone of multipliers of [a, b]: no sign that pairs with an infinite bound."""
    v = torch.where(torch.isinf(a), v.clamp(min=0), v)
    return torch.where(torch.isinf(b), v.clamp(max=0), v)


def _recession(v, a, b):
    """Onto the recession cone of [a, b]."""
    v = torch.where(torch.isinf(a), v, v.clamp(min=0))
    return torch.where(torch.isinf(b), v, v.clamp(max=0))


def _support(v, a, b):
    zero = torch.zeros_like(v)
    return (torch.where(v > 0, b * v, zero) + torch.where(v < 0, a * v, zero)).sum(0)


def _solve64(p, scaled, specs, tol, max_iter, every=64):
    """Restarted reflected Halpern PDHG on one batch, all columns at once, in 64 bits."""
    dr, dc, A, At, norm, _ = scaled
    B, eta = len(specs), 0.998 / norm
    cols = torch.arange(B, device="cuda")
    kind = torch.from_numpy(specs["kind"].astype(np.int64)).cuda()
    var = torch.from_numpy(specs["var"].astype(np.int64)).cuda()
    c, lo, hi, l, u = p.c[:, None], p.lo[:, None], p.hi[:, None], p.rl[:, None], p.ru[:, None]
    drc, dcc = dr[:, None], dc[:, None]
    bound = bool((kind == 1).all())
    if bound:
        lo, hi = lo.repeat(1, B), hi.repeat(1, B)
        lo[var, cols] = torch.maximum(p.lo[var], torch.from_numpy(specs["lo"].copy()).cuda())
        hi[var, cols] = torch.minimum(p.hi[var], torch.from_numpy(specs["hi"].copy()).cuda())
        cnorm = (dc * p.c).norm().expand(B)
    else:
        c = torch.zeros(p.n, B, dtype=torch.float64, device="cuda")
        c[var, cols] = torch.from_numpy(specs["sign"].copy()).cuda()
        cnorm = (dcc * c).norm(dim=0)
    cs, los, his, ls, us = dcc * c, lo / dcc, hi / dcc, drc * l, drc * u
    fl, fu = torch.isfinite(ls), torch.isfinite(us)
    b = torch.where(fl & fu, torch.where(ls.abs() > us.abs(), ls, us), torch.where(fl, ls, torch.where(fu, us, 0 * dr[:, None])))
    w = cnorm / b.norm()
    w = torch.where((cnorm > 0) & torch.isfinite(w) & (w > 0), w, torch.ones_like(w))
    X = torch.zeros(p.n, B, dtype=torch.float64, device="cuda").clamp(los, his)
    Y = torch.zeros(p.m, B, dtype=torch.float64, device="cuda")
    X0, Y0 = X.clone(), Y.clone()
    out = {f: torch.full((B,), math.nan, dtype=torch.float64, device="cuda") for f in _FIELDS if f not in _WHOLE}
    out["x"] = torch.zeros(B, p.n, dtype=torch.float64, device="cuda")
    out["y"] = torch.zeros(B, p.m, dtype=torch.float64, device="cuda")
    active = torch.ones(B, dtype=torch.bool, device="cuda")
    k = K = 0
    r0 = rprev = -1.0
    while True:
        L = min(every, max_iter - K)
        tau, sigma = eta / w, eta * w
        for t in range(L):
            step = tau * (cs + At @ Y)
            xh = torch.minimum(torch.maximum(X - step, los), his)
            H = A @ (2 * xh - X)
            v = Y / sigma + H
            yh = sigma * (v - v.clamp(ls, us))
            if t == L - 1:
                dx, dy = xh - X, yh - Y
            a = 1.0 / (k + t + 2)
            X = (1 - a) * (2 * xh - X) + a * X0
            Y = (1 - a) * (2 * yh - Y) + a * Y0
        # the check, at (xh, yh), in the space of the inputs
        x, y = torch.minimum(torch.maximum(dcc * xh, lo), hi), drc * yh
        ax, adx, aty = A @ xh, A @ dx, (At @ yh) / dcc
        q = c + aty
        r = _barrier(-q, lo, hi)
        pres, dres = (ax / drc - (ax / drc).clamp(l, u)).norm(dim=0), (q + r).norm(dim=0)
        rel_p, rel_d = pres / (1 + (ax / drc).norm(dim=0)), dres / (1 + c.norm(dim=0))
        dsum, ctx = _support(r, lo, hi) + _support(y, l, u), (c * x).sum(0)
        rel_g = (ctx + dsum).abs() / (1 + ctx.abs() + dsum.abs())
        res = ((w / eta) * dx.square().sum(0) + dy.square().sum(0) / (eta * w) - 2 * (dy * adx).sum(0)).clamp(min=0).sqrt()
        dyp = _barrier(dy, ls.expand_as(dy), us.expand_as(dy))
        drr = _barrier(r - _barrier(-c - aty + (At @ dy) / dcc, lo, hi), lo, hi)
        ph = _support(drc * dyp, l, u) + _support(drr, lo, hi)
        cdx = (c * dcc * dx).sum(0)
        inf_p = (ph < 0) & (((At @ dyp) / dcc + drr).norm(dim=0) <= tol * ph.abs())
        inf_d = ((cdx < 0) & ((dcc * dx - _recession(dcc * dx, lo, hi)).norm(dim=0) <= tol * cdx.abs())
                 & ((adx / drc - _recession(adx / drc, l, u)).norm(dim=0) <= tol * cdx.abs()))
        solved = ((rel_p <= tol) & (rel_d <= tol) & (rel_g <= tol)) | inf_p | inf_d
        K += L
        last = K >= max_iter
        done = active if last else active & solved
        now = {"obj": ctx, "dual_obj": -dsum, "rel_primal": rel_p, "rel_dual": rel_d, "rel_gap": rel_g,
               "safe_bound": -dsum - tol * (1 + ctx.abs() + dsum.abs())}
        for f, value in now.items():
            out[f] = torch.where(done, value.expand(B), out[f])
        out["x"][done], out["y"][done] = x.T[done], y.T[done]
        active = active & ~solved
        if last or not bool(active.any()):
            return out
        mean = float(res[active].mean())
        if r0 < 0:
            r0 = rprev = mean
        inner, total = k + L - 1, K - 1
        if mean <= 0.2 * r0 or (mean <= 0.8 * r0 and mean > rprev) or inner > 0.36 * total:
            ddx, ddy = (xh - X0).norm(dim=0), (yh - Y0).norm(dim=0)
            d = ddy / ddx
            fine = active & (ddx > 0) & (ddy > 0) & torch.isfinite(d)
            w = torch.where(fine, (0.5 * d.log() + 0.5 * w.log()).exp(), w)
            X0, Y0 = xh.clone(), yh.clone()
            X, Y, k, r0 = xh, yh, 0, mean
        else:
            k += L
        rprev = mean


def exact(case, seed):
    if case["lps"] * case["parts"] * _nnz(case) * case["iters"] > 1.5e11:
        return None  # minutes in 64 bits
    got = []
    for p, batches in _inputs(case, seed):
        scaled = _scaled(p)
        if case["call"] == "create":
            norm = scaled[4]
            return {"eta": 0.998 / norm, "norm": norm, "iters": None, "row": scaled[0], "col": scaled[1]}
        got += [_solve64(p, scaled, sp, case["tol"], case["iters"]) for sp in batches]
    out = {f: None if f in _WHOLE else torch.cat([g[f] for g in got]) for f in _FIELDS}
    if case.get("whole"):  # where a solve to a tolerance ends is its own: only its objectives are the problem's
        return {**{f: out[f] if f in ("obj", "dual_obj") else None for f in _FIELDS}, "x": None, "y": None}
    if case["call"] == "serve":
        return {**out, "x": torch.cat([g["x"] for g in got]), "y": torch.cat([g["y"] for g in got])}
    return {**out, "x": [g["x"] for g in got], "y": [g["y"] for g in got]}
