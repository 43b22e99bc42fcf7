"""GPU: the step kernels at the edges of their row groups, batches of entries,
row windows and column tiles, against the same three iterations in plain
numpy FP64 (Sec. 4, Eq. mainiter and the operator T)."""
import types

import numpy as np
import pytest

import lpgen

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lpb():
    import torch

    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2601_21990_gb300 import _build, lpb as mod

    _build.build()
    mod.load()
    return mod


def _lp(m, n, longest, seed):
    """Rows of 0 .. longest entries in turn (every remainder of a batch of
    entries, empty rows among them), box [0, 10], rows around a point."""
    rng = np.random.default_rng(seed)
    lengths = np.minimum(np.arange(m) % (longest + 1), n).astype(np.int64)
    rng.shuffle(lengths)
    cols = np.concatenate([np.sort(rng.choice(n, k, replace=False)) for k in lengths])
    ptr = np.zeros(m + 1, dtype=np.int64)
    np.cumsum(lengths, out=ptr[1:])
    x0 = rng.uniform(0.0, 10.0, n)
    lp = lpgen.LPData(m, n, ptr, cols.astype(np.int32), lpgen._signed_uniform(rng, cols.size), rng.standard_normal(n),
                      None, None, np.zeros(n), np.full(n, 10.0), x0, "steps")
    lpgen._rows_around(lp, x0, rng)
    return lp


def _three_iterations(lp, specs, dr, dc, eta, iters=3):
    rows = np.repeat(np.arange(lp.m), np.diff(lp.row_ptr))
    v = dr[rows] * lp.vals * dc[lp.col_idx]

    def a(x):
        out = np.zeros((lp.m, x.shape[1]))
        np.add.at(out, rows, v[:, None] * x[lp.col_idx])
        return out

    def at(y):
        out = np.zeros((lp.n, y.shape[1]))
        np.add.at(out, lp.col_idx, v[:, None] * y[rows])
        return out

    k = len(specs.kind)
    c = np.repeat((dc * lp.c)[:, None], k, 1)
    lo, hi = np.repeat((lp.var_lo / dc)[:, None], k, 1), np.repeat((lp.var_hi / dc)[:, None], k, 1)
    for q in range(k):
        j = specs.var[q]
        if specs.kind[q] == 1:
            lo[j, q], hi[j, q] = max(lp.var_lo[j], specs.lo[q]) / dc[j], min(lp.var_hi[j], specs.hi[q]) / dc[j]
        elif specs.kind[q] == 2:
            c[:, q] = 0.0
            c[j, q] = dc[j] * specs.sign[q]
    l, u = (dr * lp.row_lo)[:, None], (dr * lp.row_hi)[:, None]
    b = np.where(np.abs(l) > np.abs(u), l, u)
    w = np.linalg.norm(c, axis=0) / np.linalg.norm(b)
    tau, sigma = eta / w, eta * w
    x, y = np.clip(np.zeros_like(c), lo, hi), np.zeros((lp.m, k))
    x0, y0 = x, y
    for t in range(iters):
        xh = np.clip(x - tau * (c + at(y)), lo, hi)
        xb = 2 * xh - x
        s = y / sigma + a(xb)
        yh = sigma * (s - np.clip(s, l, u))
        x = (t + 1) / (t + 2) * xb + x0 / (t + 2)
        y = (t + 1) / (t + 2) * (2 * yh - y) + y0 / (t + 2)
    return (dc[:, None] * xh).T, (dr[:, None] * yh).T


def _specs(lp, k, seed):
    rng = np.random.default_rng(seed)
    var = rng.integers(0, lp.n, k)
    kind = np.arange(k) % 3  # base LP, a box, an objective
    return types.SimpleNamespace(kind=kind, var=var, lo=rng.uniform(1.0, 3.0, k), hi=rng.uniform(4.0, 9.0, k),
                                 sign=np.where(rng.random(k) < 0.5, 1.0, -1.0))


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("m,n,longest,lps", [
    (37, 50, 9, 1), (60, 41, 32, 2), (100, 90, 33, 3), (100, 90, 33, 5), (200, 300, 40, 9), (300, 200, 31, 17),
    (2047, 700, 12, 33), (2048, 900, 33, 64), (2049, 4097, 34, 65), (4100, 2100, 17, 129), (700, 900, 300, 40),
])
def test_steps_match_plain_iterations(lpb, precision, m, n, longest, lps):
    """x^ and y^ after three iterations.  The batch runs the kernels of every
    row-group width, grids of less and of more than one wave, rows of one and
    of several segments.  FP32 tolerance: a sum of k <= 41 products (longer
    rows are cut into pieces of at most 75) is off by at most k u |a||x|, and
    |a||x| <= sqrt(k) times the norms; six products: 6 * 75^1.5 u < 4000 u of
    the largest value.  FP64: the same with its u, times 4 for the oracle's own
    rounding."""
    lp = _lp(m, n, longest, m + lps)
    sp = _specs(lp, lps, lps)
    h = lpb.Handle(lp, precision=lpb.FP64 if precision == "fp64" else lpb.MIXED)
    dr, dc = h.scaling()
    ex, ey = _three_iterations(lp, sp, dr, dc, h.info()[0])
    u = 2.0 ** -53 * 4 if precision == "fp64" else 2.0 ** -24
    specs = lpb.specs_array(sp.kind, sp.var, sp.lo, sp.hi, sp.sign)
    for _ in range(2):  # a captured interval and its replay
        b = h.solve(specs, tol=1e-12, max_iter=3)
        assert (b.results()["iters"] == 3).all()
        for q in range(lps):
            _, x, y = b.result(q)
            assert np.abs(x - ex[q]).max() <= 4000 * u * max(1.0, np.abs(ex[q] / dc).max()) * dc.max(), q
            assert np.abs(y - ey[q]).max() <= 4000 * u * max(1.0, np.abs(ey[q] / dr).max()) * dr.max(), q
        b.free()
    h.close()


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("m,n,longest,lps", [
    (1500, 3000, 600, 1), (1500, 3000, 600, 2), (1500, 3000, 600, 3), (1500, 3000, 600, 5), (1500, 3000, 600, 8),
    (700, 3000, 257, 4), (400, 3000, 600, 1), (5000, 900, 40, 2)])
def test_narrow_batches_match_plain_iterations(lpb, precision, m, n, longest, lps):
    """One and two lanes a row: long rows of more and of fewer segments than
    four waves of SMs, the last block of segments not full, and short rows in
    the narrow order.  A segment is cut into 64 or 128 pieces of at most four
    entries, so k <= 4 + 127 + 2 + 5 additions follow one another in a row of
    600, and |a||x| <= sqrt(600) times the norms; six products:
    6 * 138 * 24.5 u < 20400 u of the largest value (FP64: times 4)."""
    lp = _lp(m, n, longest, m + lps)
    sp = _specs(lp, lps, lps)
    h = lpb.Handle(lp, precision=lpb.FP64 if precision == "fp64" else lpb.MIXED)
    dr, dc = h.scaling()
    ex, ey = _three_iterations(lp, sp, dr, dc, h.info()[0])
    u = 2.0 ** -53 * 4 if precision == "fp64" else 2.0 ** -24
    b = h.solve(lpb.specs_array(sp.kind, sp.var, sp.lo, sp.hi, sp.sign), tol=1e-12, max_iter=3)
    for q in range(lps):
        _, x, y = b.result(q)
        assert np.abs(x - ex[q]).max() <= 20400 * u * max(1.0, np.abs(ex[q] / dc).max()) * dc.max(), q
        assert np.abs(y - ey[q]).max() <= 20400 * u * max(1.0, np.abs(ey[q] / dr).max()) * dr.max(), q
    b.free()
    h.close()


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("lps", [7, 8, 31, 33, 40])
def test_points_of_many_columns_equal_those_of_one(lpb, precision, lps):
    """A batch's points, extracted together (tiles from 8 columns on), are bit
    for bit those of each LP solved alone (one column); an LP with an empty
    box among them has zeros.  One check, so no restart couples the LPs."""
    lp = _lp(130, 97, 6, 3)
    sp = _specs(lp, lps, lps)
    sp.kind[3], sp.lo[3], sp.hi[3] = 1, 5.0, 4.0  # an empty box
    specs = lpb.specs_array(sp.kind, sp.var, sp.lo, sp.hi, sp.sign)
    h = lpb.Handle(lp, precision=lpb.FP64 if precision == "fp64" else lpb.MIXED)
    b = h.solve(specs, tol=1e-12, max_iter=64)
    for q in range(lps):
        r, x, y = b.result(q)
        if q == 3:
            assert r.status == lpb.PRIMAL_INFEASIBLE and not x.any() and not y.any()
            continue
        one = h.solve(specs[q:q + 1], tol=1e-12, max_iter=64)
        _, x1, y1 = one.result(0)
        assert np.array_equal(x, x1) and np.array_equal(y, y1), q
        one.free()
    b.free()
    h.close()


@pytest.mark.parametrize("precision", ["fp64", "mixed", "polish"])
@pytest.mark.parametrize("m,n,longest,lps", [
    (1, 3, 1, 1), (37, 50, 9, 2), (60, 41, 32, 7), (100, 90, 60, 33), (200, 300, 40, 150), (150, 100, 300, 170),
    (64, 700, 500, 5), (300, 200, 12, 400),
])
def test_resident_intervals_equal_the_steps(lpb, precision, m, n, longest, lps):
    """Small matrices run whole intervals in one launch; timed solves
    (profile = 1) run the step kernels.  Every result and point is bit for bit
    the same: one, two and four columns a block, ragged tiles, empty and long
    rows, boxes and objectives, several intervals and a short last one."""
    lp = _lp(m, n, longest, m + lps)
    sp = _specs(lp, lps, lps)
    specs = lpb.specs_array(sp.kind, sp.var, sp.lo, sp.hi, sp.sign)
    opts = dict(precision=lpb.FP64 if precision == "fp64" else lpb.MIXED)
    if precision == "polish":
        opts["polish_stall_checks"] = 1
    got = []
    for profile in (0, 1):
        h = lpb.Handle(lp, profile=profile, **opts)
        for _ in range(2 - profile):  # a captured interval and its replay
            b = h.solve(specs, tol=1e-9, max_iter=200)
            kernels, steps = b.profile().kernels, sum(b.profile().launches[:2])
            got.append([b.results()] + [v for q in range(lps) for v in b.result(q)[1:]])
            b.free()
        assert kernels > steps if profile else lp.nnz == 0 or lp.nnz > 1500 or kernels < steps, (kernels, steps)
        h.close()
    for other in got[1:]:
        assert all(np.array_equal(x, y, equal_nan=x.dtype.kind == "f") if x.dtype.names is None
                   else all(np.array_equal(x[f], y[f], equal_nan=x[f].dtype.kind == "f") for f in x.dtype.names)
                   for x, y in zip(got[0], other))


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("thr", [1, 32, 2 ** 31 - 1])
@pytest.mark.parametrize("m,n,longest,lps", [(130, 90, 60, 3), (300, 200, 60, 9), (2050, 900, 24, 40)])
def test_steps_at_every_long_row_threshold(lpb, precision, thr, m, n, longest, lps):
    """From a block for almost every row to none for any (the largest
    threshold), on row counts that are no whole windows: x^ and y^ after three
    iterations, as plain iterations give them.  Tolerance: a sum of k products,
    k at most the longest row or column, is off by k u sqrt(k) times the norms;
    six products: 6 k^1.5 u of the largest value; FP64 the same with its u,
    times 4 for the oracle's own rounding."""
    lp = _lp(m, n, longest, m + lps)
    sp = _specs(lp, lps, lps)
    h = lpb.Handle(lp, precision=lpb.FP64 if precision == "fp64" else lpb.MIXED, profile=1)
    t = h.tuning()
    t.long_row_primal = t.long_row_dual = thr
    h.set_tuning(t)
    assert (h.tuning().long_row_primal, h.tuning().long_row_dual) == (thr, thr)
    dr, dc = h.scaling()
    ex, ey = _three_iterations(lp, sp, dr, dc, h.info()[0])
    k = max(np.diff(lp.row_ptr).max(), np.bincount(lp.col_idx, minlength=n).max())
    tol = 6 * k ** 1.5 * (2.0 ** -53 * 4 if precision == "fp64" else 2.0 ** -24)
    b = h.solve(lpb.specs_array(sp.kind, sp.var, sp.lo, sp.hi, sp.sign), tol=1e-12, max_iter=3)
    for q in range(lps):
        _, x, y = b.result(q)
        assert np.abs(x - ex[q]).max() <= tol * max(1.0, np.abs(ex[q] / dc).max()) * dc.max(), q
        assert np.abs(y - ey[q]).max() <= tol * max(1.0, np.abs(ey[q] / dr).max()) * dr.max(), q
    b.free()
    h.close()


def test_packed_rows_take_no_room_for_long_rows(lpb):
    """A handle holds each entry once per orientation in the forms that the
    checks and the long rows read (FP64, FP32, its low part, double-float, a
    column: 28 bytes), and again only where it stands in a short row.  Here
    all but 64 of eight million entries stand in rows and columns of 40 and
    more: 56 bytes an entry, a generous 400 bytes a row or column, and 64 MB."""
    import torch

    m, n, dense = 72, 200_000, 40
    lengths = np.array([n] * dense + [2] * (m - dense), dtype=np.int64)
    ptr = np.concatenate([[0], np.cumsum(lengths)])
    rng = np.random.default_rng(0)
    cols = np.concatenate([np.tile(np.arange(n), dense), np.arange(2 * (m - dense))]).astype(np.int32)
    lp = lpgen.LPData(m, n, ptr, cols, lpgen._signed_uniform(rng, cols.size), np.ones(n), np.full(m, -1.0), np.ones(m),
                      np.zeros(n), np.ones(n), np.zeros(n), "dense_rows")
    lpb.Handle(_lp(37, 50, 9, 1), precision=lpb.MIXED).close()  # the context and the library's own memory
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    h = lpb.Handle(lp, precision=lpb.MIXED, ruiz_iters=1, power_max_iter=2)
    torch.cuda.synchronize()
    held = before - torch.cuda.mem_get_info()[0]
    h.close()
    assert 56 * cols.size <= held <= 56 * cols.size + 400 * (m + n) + (64 << 20), held


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_tune_batch_times_the_kernel_that_a_solve_runs(lpb, precision):
    """On a small matrix a solve runs whole intervals in one launch, in well
    under the time of its steps one by one: lpb_tune_batch reports that kernel,
    and the step kernels on a handle whose solves time them (profile = 1)."""
    lp = _lp(200, 400, 20, 7)
    opts = dict(precision=lpb.FP64 if precision == "fp64" else lpb.MIXED)
    us = {}
    for profile in (0, 1):
        h = lpb.Handle(lp, profile=profile, **opts)
        sp = _specs(lp, 16, 0)
        b = h.solve(lpb.specs_array(sp.kind, sp.var, sp.lo, sp.hi, sp.sign), tol=1e-12, max_iter=128)
        p = b.profile()
        assert (p.kernels < sum(p.launches[:2])) == (profile == 0)
        us[profile] = h.tune_batch([16])[0][0]
        if profile:
            steps = 1e3 * (p.ms[0] + p.ms[1]) / p.launches[0]
        b.free()
        h.close()
    assert us[0] < 0.85 * us[1] and us[0] < 0.85 * steps, (us, steps)


@pytest.mark.parametrize("lps,lanes", [(3, 1), (7, 2), (13, 4), (30, 8)])
def test_row_orders_agree_on_a_large_matrix(lpb, lps, lanes):
    """Narrow batches take the rows as they stand, wider ones by length, and at
    eight lanes the primal step of a matrix whose points exceed L2 the former:
    bit for bit the same points and results, as a short row is summed in its
    own order whoever takes it.  64 LPs (16 lanes, by length) against the first
    of them alone; one check, so no restart couples them."""
    m, n = 150_000, 600_000
    rng = np.random.default_rng(1)
    lengths = rng.integers(0, 9, m)
    ptr = np.concatenate([[0], np.cumsum(lengths)]).astype(np.int64)
    cols = np.concatenate([np.sort(c) for c in np.split(rng.integers(0, n, ptr[-1]), ptr[1:-1])]).astype(np.int32)
    x0 = rng.uniform(0.0, 10.0, n)
    lp = lpgen.LPData(m, n, ptr, cols, lpgen._signed_uniform(rng, cols.size), rng.standard_normal(n), None, None,
                      np.zeros(n), np.full(n, 10.0), x0, "orders")
    lpgen._rows_around(lp, x0, rng)
    sp = _specs(lp, 64, 3)
    specs = lpb.specs_array(sp.kind, sp.var, sp.lo, sp.hi, sp.sign)
    h = lpb.Handle(lp, precision=lpb.MIXED, power_max_iter=50)
    wide = h.solve(specs, tol=1e-12, max_iter=64)
    narrow = h.solve(specs[:lps], tol=1e-12, max_iter=64)
    assert np.array_equal(wide.results()[:lps], narrow.results())
    for q in (0, lps // 2, lps - 1):
        for a, b in zip(wide.result(q)[1:], narrow.result(q)[1:]):
            assert np.array_equal(a, b), q
    wide.free(), narrow.free()
    h.close()


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("lps", [1, 5, 200, 1500])
def test_points_of_empty_boxes_are_zero_among_others(lpb, precision, lps):
    """LPs whose box is empty end at admission, with zeros for their points;
    the others' points are those of the same LPs without them.  One check, so
    no restart couples the LPs."""
    lp = _lp(40, 300, 6, 3)
    sp = _specs(lp, lps, lps)
    sp.kind = np.where(np.arange(lps) % 3 == 0, 1, sp.kind)
    empty = np.arange(lps) % 3 == 0
    sp.lo, sp.hi = np.where(empty, 5.0, sp.lo), np.where(empty, 4.0, sp.hi)
    specs = lpb.specs_array(sp.kind, sp.var, sp.lo, sp.hi, sp.sign)
    h = lpb.Handle(lp, precision=lpb.FP64 if precision == "fp64" else lpb.MIXED)
    junk = h.solve(lpb.specs_array(np.zeros(lps, int), sp.var), tol=1e-12, max_iter=64)  # (memory with points in it)
    junk.free()
    b = h.solve(specs, tol=1e-12, max_iter=64)
    assert (b.results()["status"][empty] == lpb.PRIMAL_INFEASIBLE).all()
    rest = np.flatnonzero(~empty)
    alone = h.solve(specs[rest], tol=1e-12, max_iter=64) if rest.size else None
    for q in range(lps):
        _, x, y = b.result(q)
        if empty[q]:
            assert not x.any() and not y.any(), q
        else:
            _, x1, y1 = alone.result(int(np.searchsorted(rest, q)))
            assert np.array_equal(x, x1) and np.array_equal(y, y1), q
    b.free()
    h.close()
