"""The kernel that keeps the pivots instead of a tableau, and the tableau kernel's deferred
updates in Phase I (the planner's choices under the largest-coefficient rule), against the
kernels that update a tableau after every pivot, and against the oracle.

Both form every tableau value by the same operations in the same order, so statuses, pivot
counts and bases are equal, bit for bit; the FP64 results, which are read straight off, are
too.  Refined FP32 results differ in the rounding of a correction of order 1e-7 times the
values, and in plain FP32 mode not at all."""
import ctypes

import numpy as np
import pytest
import torch

import oracle
import synth
from lp_helpers import compare, host, to_device

pytestmark = pytest.mark.gpu

GMEM, REG, PACK, WARP = 2, 3, 4, 5


@pytest.fixture(scope="module")
def solver():
    from paper_1609_08114_gb300 import Solver
    return Solver(0)


def _batch(sb, dtype):
    from paper_1609_08114_gb300 import LPBatch
    return LPBatch.from_packed(sb.m, sb.n, sb.A, sb.b, sb.c, device="cuda", dtype=dtype)


# One warp per LP up to 32 and 64 rows or columns, two up to 128, four up to 256, eight
# beyond: both sides of each edge, one row or column, odd sizes.
SHAPES = [(33, 1), (1, 33), (32, 33), (40, 64), (64, 65), (65, 40), (97, 101), (127, 127), (127, 3), (128, 20),
          (20, 128), (129, 129), (255, 30), (256, 257), (300, 41)]


@pytest.mark.parametrize("m,n", SHAPES)
@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("prec", ["fp64", "fp32_refine", "fp32"])
def test_same_pivots_as_the_full_update(solver, m, n, dtype, prec):
    sb = synth.type1(60, m, n, seed=m + 1000 * n)
    batch = _batch(sb, dtype)
    if prec == "fp64" or max(m, n) > 127:
        full = GMEM
    else:      # the kernel that has this size and type when a kernel is asked for
        full = WARP if dtype == torch.float64 and m * n <= 10000 else REG
    got, ref = host(solver.solve(batch, prec=prec)), host(solver.solve(batch, prec=prec, kernel=full))
    for name in ("status", "iters", "basis"):
        assert np.array_equal(got[name], ref[name]), name
    if prec == "fp32_refine":
        for name in ("obj", "x", "y"):
            np.testing.assert_allclose(got[name], ref[name], rtol=0, atol=1e-9)
    else:
        for name in ("obj", "x", "y"):
            assert np.array_equal(got[name], ref[name]), name
    if dtype == torch.float64 and prec == "fp32_refine":
        compare(sb, got, obj_rtol=1e-8)
    assert solver.sync_error() == 0


# LPs that would share a warp (two of up to 15, one of up to 31 rows and columns), enough of
# them to leave the kernel that does so.
@pytest.mark.parametrize("m,n", [(8, 1), (1, 8), (9, 15), (15, 15), (16, 16), (1, 31), (31, 1), (20, 27), (31, 31)])
@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
def test_same_pivots_as_several_lps_per_warp(solver, m, n, dtype):
    sb = synth.type1(20001, m, n, seed=m + 1000 * n)
    batch = _batch(sb, dtype)
    got, ref = host(solver.solve(batch, prec="fp32")), host(solver.solve(batch, prec="fp32", kernel=PACK))
    for name in ("status", "iters", "basis", "obj", "x", "y"):
        assert np.array_equal(got[name], ref[name]), name


@pytest.mark.parametrize("m,n", [(40, 33), (64, 64), (130, 30)])
@pytest.mark.parametrize("dtype,prec", [(torch.float32, "fp32"), (torch.float32, "fp32_refine"), (torch.float64, "fp64")])
def test_same_pivots_under_the_random_rule(solver, m, n, dtype, prec):
    """In a batch that fills the GPU (smaller ones keep the full update under this rule)."""
    sb = synth.type1(2500, m, n, seed=m + 31 * n)
    batch = _batch(sb, dtype)
    full = GMEM if prec == "fp64" or max(m, n) > 127 else REG
    got = host(solver.solve(batch, prec=prec, pivot_rule="rpc", seed=11))
    ref = host(solver.solve(batch, prec=prec, pivot_rule="rpc", seed=11, kernel=full))
    for name in ("status", "iters", "basis"):
        assert np.array_equal(got[name], ref[name]), name
    np.testing.assert_allclose(got["obj"], ref["obj"], rtol=1e-9)
    assert solver.sync_error() == 0


def _boxed(count, m, n, seed):
    """LPs of many pivots: rows of both signs and a bound on every variable."""
    r = np.random.default_rng(seed)
    return synth.pack([(np.vstack([r.normal(size=(m - n, n)), np.eye(n)]), r.uniform(1, 5, size=m),
                        r.uniform(0.1, 1, size=n)) for _ in range(count)])


@pytest.mark.parametrize("m,n", [(60, 25), (100, 45), (180, 70)])
@pytest.mark.parametrize("prec,rtol", [("fp64", 1e-9), ("fp32_refine", 1e-8)])
def test_more_pivots_than_the_history_holds(solver, m, n, prec, rtol):
    """Pivots beyond the shared-memory history (in the workspace slot) and beyond the most
    the kernel takes (such LPs go to the tableau kernel)."""
    sb = _boxed(80, m, n, seed=m)
    got = host(solver.solve(to_device(sb), prec=prec))
    ref = oracle.solve_batch(sb)
    assert ref["iters"].max() > 12
    assert np.array_equal(got["status"], ref["status"])
    ok = ref["status"] == 0
    assert np.all(np.abs(got["obj"] - ref["obj"])[ok] <= rtol * (1 + np.abs(ref["obj"][ok])))
    if prec == "fp64":
        assert np.array_equal(got["iters"], ref["iters"])
    assert solver.sync_error() == 0


# Both sides of the deferred updates' least size, of 128 and 256 rows or columns (the CTA's
# threads), and of a row's last vector; pivots from fewer than wait at once to many sweeps.
@pytest.mark.parametrize("m,n", [(30, 38), (33, 41), (60, 20), (64, 64), (90, 97), (128, 60), (60, 131), (200, 200),
                                 (258, 30), (30, 259)])
@pytest.mark.parametrize("prec", ["fp32", "fp32_refine"])
def test_deferred_updates_in_phase_one(solver, m, n, prec):
    """Two-phase LPs (infeasible and unbounded ones among them): the same pivots, statuses
    and bases as with a full update after every pivot."""
    sb = synth.type2(80, m, n, seed=m + n, frac_infeasible=0.1, frac_unbounded=0.1)
    batch = to_device(sb)
    got = host(solver.solve(batch, prec=prec))
    ref = host(solver.solve(batch, prec=prec, kernel=GMEM))
    for name in ("status", "iters", "basis"):
        assert np.array_equal(got[name], ref[name]), name
    for name in ("obj", "x", "y"):
        if prec == "fp32":
            assert np.array_equal(got[name], ref[name], equal_nan=True), name
        else:
            fin = np.isfinite(ref[name])
            assert np.array_equal(got[name][~fin], ref[name][~fin])
            np.testing.assert_allclose(got[name][fin], ref[name][fin], rtol=1e-9, atol=1e-9)
    assert solver.sync_error() == 0


@pytest.mark.parametrize("m,n", [(50, 40), (140, 30)])
@pytest.mark.parametrize("prec", ["fp64", "fp32_refine"])
def test_what_it_does_not_take(solver, m, n, prec):
    """Non-finite data, values beyond FP32, negative right-hand sides, zero rows and columns."""
    sb = synth.type1(12, m, n, seed=5)
    A, b, c = sb.A.reshape(12, m, n), sb.b.reshape(12, m), sb.c.reshape(12, n)
    A[0, m - 1, n - 1], A[1, 0, 0], b[2, 1], c[3, 2] = np.nan, np.inf, np.nan, -np.inf
    A[4, 3, 3] = 1e39                    # beyond FP32: FP64 solves it
    b[5, 7] = -0.5                       # infeasible: A > 0
    A[6, :, 4] = 0.0                     # a zero column with a positive cost: unbounded
    c[7] = -1.0                          # optimal at the origin, no pivot
    A[8, 2], b[9, 3] = 0.0, 0.0
    got = host(solver.solve(to_device(sb), prec=prec))
    want = [4, 4, 4, 4, None, 1, 2, 0, 0, 0, 0, 0]
    for k, w in enumerate(want):
        if w is not None:
            assert got["status"][k] == w, k
    assert got["iters"][7] == 0 and got["obj"][7] == 0.0
    assert solver.sync_error() == 0


def test_less_workspace_than_its_slots(solver):
    """A workspace without room for the history slots: the kernels that need none."""
    from paper_1609_08114_gb300 import _lib
    sb = synth.type1(3000, 100, 90, seed=3)
    batch = _batch(sb, torch.float64)
    want = host(solver.solve(batch))
    out, opt = solver.alloc_result(batch), solver.options("fp32_refine")
    cb, cr = batch.cstruct(), out.cstruct()
    full = solver.workspace_size(batch, opt)
    ws = torch.empty(full - 256, dtype=torch.uint8, device="cuda")
    stream = ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)
    call = lambda size: solver.lib.lpb_solve(  # noqa: E731
        solver.h, ctypes.byref(cb), ctypes.byref(opt), ctypes.byref(cr), ctypes.c_void_p(ws.data_ptr()), size, stream)
    assert call(full - 256) == _lib.OK
    got = host(out)
    for name in ("status", "iters", "basis"):
        assert np.array_equal(got[name], want[name]), name
    assert call(256) == _lib.ENOMEM


@pytest.mark.parametrize("m,n", [(12, 9), (31, 33), (64, 65), (65, 30), (100, 100), (127, 21)])
@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("turn", [None, 1e-3])
def test_objectives_of_one_polytope(solver, m, n, dtype, turn):
    """Warm starts (directions that turn slowly) and cold ones (independent directions, a
    last chunk that is not full) against FP64 solves of the same objectives."""
    r = np.random.default_rng(m + n)
    A, b, _ = synth.type1(1, m, n, seed=m).lp(0)
    count = 16 * 40 + 5
    C = r.normal(size=(count, n)) if turn is None else (
        r.uniform(0, 1, size=n)[None] + turn * np.arange(count)[:, None] * r.normal(size=n)[None])
    args = [torch.tensor(v, device="cuda", dtype=dtype) for v in (A, b, C)]
    got = host(solver.solve_shared(*args, prec="fp32_refine"))
    ref = host(solver.solve_shared(*[a.double() for a in args], prec="fp64"))
    assert np.array_equal(got["status"], ref["status"])
    assert np.all(np.abs(got["obj"] - ref["obj"]) <= 1e-8 * (1 + np.abs(ref["obj"])))
    if turn is not None:
        assert got["iters"].mean() < 0.5 * ref["iters"].mean()
    assert solver.sync_error() == 0
