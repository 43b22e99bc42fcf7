"""GPU: the resident interval kernel (csrc/lpb_resident.cu) where rows are cut:
rows of A and of its transpose of one, two and three segments, at one, two and
four columns a block with ragged last tiles, alone and in a joint solve.  That
kernel is shown to have run (a solve of it launches fewer kernels than it takes
steps), and its results are bit for bit those of the step kernels, which run
when a solve times its steps (profile = 1)."""
import numpy as np
import pytest

import lpgen

pytestmark = pytest.mark.gpu

# past the long-row threshold of 32, and about and past the 256 entries of a segment
LENGTHS = [600, 513, 300, 257, 256, 60, 33, 32]


@pytest.fixture(scope="module")
def lpb():
    import torch

    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    from paper_2601_21990_gb300 import _build, lpb as mod

    _build.build()
    mod.load()
    return mod


def _lp(long_side, seed):
    """64 rows on 700 columns, the first of LENGTHS entries, the others of 0 to
    8; or its transpose, whose columns are those."""
    rng = np.random.default_rng(seed)
    a = np.zeros((64, 700))
    for i, k in enumerate(LENGTHS + [q % 9 for q in range(64 - len(LENGTHS))]):
        a[i, rng.choice(700, k, replace=False)] = lpgen._signed_uniform(rng, k)
    if long_side == "columns":
        a = a.T.copy()
    m, n = a.shape
    x0 = rng.uniform(0.0, 10.0, n)
    slack = rng.uniform(0.0, 1.0, m)
    return lpgen.from_dense(a, rng.standard_normal(n), a @ x0 - slack, a @ x0 + slack, np.zeros(n), np.full(n, 10.0))


def _specs(lpb, lp, k, seed):
    rng = np.random.default_rng(seed)
    var = rng.integers(0, lp.n, k)
    return lpb.specs_array(np.arange(k) % 3, var, rng.uniform(1.0, 3.0, k), rng.uniform(4.0, 9.0, k),
                           np.where(rng.random(k) < 0.5, 1.0, -1.0))


def _take(b, lps):
    p = b.profile()
    out = [b.results()] + [v for q in range(lps) for v in b.result(q)[1:]]
    b.free()
    return out, int(p.kernels), int(sum(p.launches[:2]))


def _same(x, y):
    if x.dtype.names is not None:
        return all(_same(x[f], y[f]) for f in x.dtype.names)
    return np.array_equal(x, y, equal_nan=x.dtype.kind == "f")


# at most 152 tiles: four columns a block only in FP32
CASES = [(p, k) for p in ("fp64", "mixed", "polish") for k in (1, 3, 5, 34, 151, 201, 303)] + \
        [("mixed", k) for k in (305, 401, 607)]


@pytest.mark.parametrize("long_side", ["rows", "columns"])
@pytest.mark.parametrize("precision,lps", CASES)
def test_cut_rows_equal_the_steps(lpb, precision, lps, long_side):
    lp = _lp(long_side, lps)
    opts = dict(precision=lpb.FP64 if precision == "fp64" else lpb.MIXED)
    if precision == "polish":
        opts["polish_stall_checks"] = 1
    specs = _specs(lpb, lp, lps, lps)
    h = lpb.Handle(lp, **opts)
    got, kernels, steps = _take(h.solve(specs, tol=1e-9, max_iter=200), lps)
    # (in FP64 the short pieces of one and two lanes are the step kernels' case)
    assert (kernels > steps) if precision == "fp64" and lps <= 4 else (kernels < steps), (kernels, steps)
    h.close()
    h = lpb.Handle(lp, profile=1, **opts)
    want, kernels, steps = _take(h.solve(specs, tol=1e-9, max_iter=200), lps)
    assert kernels > steps, (kernels, steps)
    h.close()
    assert all(_same(x, y) for x, y in zip(got, want))


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
@pytest.mark.parametrize("widths", [(5, 34, 12), (100, 33, 70)])
def test_joint_solve_of_cut_rows_equals_the_steps(lpb, precision, widths):
    lps = [_lp(side, 50 + i) for i, side in enumerate(("rows", "columns", "rows"))]
    opts = dict(precision=lpb.FP64 if precision == "fp64" else lpb.MIXED)
    specs = [_specs(lpb, lp, k, k) for lp, k in zip(lps, widths)]
    hs = [lpb.Handle(lp, **opts) for lp in lps]
    joint = [_take(b, k) for b, k in zip(lpb.Handle.solve_multi(hs, specs, tol=1e-9, max_iter=200), widths)]
    for h in hs:
        h.close()
    for lp, sp, k, (got, kernels, steps) in zip(lps, specs, widths, joint):
        assert kernels < steps, (kernels, steps)
        h = lpb.Handle(lp, profile=1, **opts)
        want, kernels, steps = _take(h.solve(sp, tol=1e-9, max_iter=200), k)
        assert kernels > steps, (kernels, steps)
        h.close()
        assert all(_same(x, y) for x, y in zip(got, want))
