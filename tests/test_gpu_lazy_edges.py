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
