"""The kernel that keeps the pivots, where it can go wrong: values that pass from one lane to
another, many LPs per CTA, many pivots, its largest configurations, little scratch."""
import numpy as np
import pytest
import torch

import synth
from lp_helpers import host, to_device

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def solver():
    from paper_1609_08114_gb300 import Solver
    return Solver(0)


@pytest.mark.parametrize("m,n", [(33, 1), (32, 33), (48, 37), (64, 64), (100, 90)])
@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
def test_refined_values_are_those_of_the_objective(solver, m, n, dtype):
    """Several LPs per CTA.  The objective is summed from the corrected x before other lanes
    read x and write it out: c.x of what was written is that sum but for FP64 rounding (1e-12
    covers some hundred operations of 2^-53, and the tableau's for an LP solved again in
    FP64).  b.y agrees to the certificate's 1e-9, where an uncorrected y is off by FP32
    rounding."""
    count = 6000
    sb = synth.type1(count, m, n, seed=m * 7 + n)
    got = host(solver.solve(to_device(sb, dtype), prec="fp32_refine"))
    assert (got["status"] == 0).all()
    t = np.float32 if dtype == torch.float32 else np.float64
    b, c = (v.astype(t).astype(np.float64) for v in (sb.b.reshape(count, m), sb.c.reshape(count, n)))
    x, y = got["x"].reshape(count, n), got["y"].reshape(count, m)
    size = np.abs(c * x).sum(axis=1)
    assert np.all(np.abs((c * x).sum(axis=1) - got["obj"]) <= 1e-12 * (1 + size))
    size = np.abs(b * y).sum(axis=1)
    assert np.all(np.abs((b * y).sum(axis=1) - got["obj"]) <= 1e-9 * (1 + np.abs(got["obj"])) + 1e-12 * size)
    assert solver.sync_error() == 0


@pytest.mark.parametrize("m,n,lo", [(130, 30, 0.1), (200, 100, -0.5), (150, 160, 0.1), (300, 257, 0.1)])
def test_refinement_ends_on_fp64_residuals(solver, m, n, lo):
    """Above 127 rows or columns corrections go on until the residuals b - A x of the binding
    rows and A^T y - c of the basic columns are 1000 times below the certificate's bar
    1e-9 (1 + max|b|) and 1e-9 (1 + max|c|) (three corrections at most, of six digits each).
    They are formed here in extended precision; FP64 adds at most n + 2 roundings of the sums."""
    count = 600
    r = np.random.default_rng(m + n)
    A, b, c = r.uniform(lo, 1, (count, m, n)), r.uniform(1, 10, (count, m)), r.uniform(0, 1, (count, n))
    if lo < 0:                   # a bound on every variable
        A[:, m - n:] = np.eye(n)
    sb = synth.pack([(A[k], b[k], c[k]) for k in range(count)])
    got = host(solver.solve(to_device(sb), prec="fp32_refine"))
    resolved = solver.stats()["resolved_fp64"]
    assert (got["status"] == 0).all() and resolved <= count // 100
    x, y = got["x"].reshape(count, n).astype(np.longdouble), got["y"].reshape(count, m).astype(np.longdouble)
    basis, over = got["basis"].reshape(count, m), 0
    for k in range(count):
        rows = np.setdiff1d(np.arange(m), basis[k][basis[k] >= n] - n)
        cols = basis[k][basis[k] < n]
        rp, rd = np.abs(b[k] - A[k] @ x[k])[rows], np.abs(y[k] @ A[k] - c[k])[cols]
        tp = 1e-12 * (1 + b[k].max()) + (n + 2) * 2.0 ** -53 * float((np.abs(A[k]) @ np.abs(x[k])).max())
        td = 1e-12 * (1 + c[k].max()) + (m + 2) * 2.0 ** -53 * float((np.abs(y[k]) @ np.abs(A[k])).max())
        over += rp.max(initial=0) > tp or rd.max(initial=0) > td
    assert over <= resolved
