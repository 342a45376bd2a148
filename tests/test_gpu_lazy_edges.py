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


GMEM, REG, PACK, WARP = 2, 3, 4, 5


def _many_pivots(count, m, n, seed, sparse=False):
    """LPs with b > 0 whose pivots are of the order of min(m, n): rows of both signs, or one
    entry in ten."""
    r = np.random.default_rng(seed)
    A = r.uniform(0.1, 1, (count, m, n)) * (r.random((count, m, n)) < 0.1) if sparse else r.normal(0.3, 1, (count, m, n))
    return synth.pack([(A[k], r.uniform(1, 10, m), r.uniform(0, 1, n)) for k in range(count)])


# One, two, four and eight warps per LP; LPs that leave the history once and several times;
# row blocks that are not full; more LPs than CTAs.
MANY = [(60, 33, 31), (3000, 40, 40), (60, 64, 63), (60, 97, 100), (60, 127, 120), (60, 61, 127), (60, 140, 30),
        (40, 200, 100), (40, 129, 257), (20, 300, 201)]


@pytest.mark.parametrize("count,m,n", MANY)
@pytest.mark.parametrize("prec,dtype", [("fp64", torch.float64), ("fp64", torch.float32), ("fp32", torch.float64),
                                        ("fp32", torch.float32), ("fp32_refine", torch.float64),
                                        ("fp32_refine", torch.float32)])
@pytest.mark.parametrize("sparse", [False, True])
def test_many_pivots_as_the_full_update(solver, count, m, n, prec, dtype, sparse):
    """Pivots applied to the tableau in between: the same operations on every value, so the same
    pivots and, where results are read straight off, the same bits.  (Refined: an LP whose
    certificate one rounding of the correction just passes and another does not is solved
    again, with pivots of its own: one in fifty is left out.)"""
    sb = _many_pivots(count, m, n, 31 * m + n, sparse)
    batch = to_device(sb, dtype)
    full = GMEM if prec == "fp64" or max(m, n) > 127 else WARP if dtype == torch.float64 and m * n <= 10000 else REG
    got, ref = host(solver.solve(batch, prec=prec)), host(solver.solve(batch, prec=prec, kernel=full))
    assert np.array_equal(got["status"], ref["status"])
    assert ref["iters"].max() > 8 + m * n // (m + n) or prec == "fp32_refine"
    if prec == "fp32_refine":
        same = (got["iters"] == ref["iters"]) & (got["basis"] == ref["basis"]).reshape(count, m).all(axis=1)
        assert (~same).sum() <= count // 50
        ok = ref["status"] == 0
        assert np.all(np.abs(got["obj"][ok] - ref["obj"][ok]) <= 1e-8 * (1 + np.abs(ref["obj"][ok])))
    else:
        for name in ("iters", "basis", "obj", "x", "y"):
            assert np.array_equal(got[name], ref[name], equal_nan=name == "obj"), name
    assert solver.sync_error() == 0


@pytest.mark.parametrize("m,n", [(31, 31), (20, 29)])
@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
def test_many_pivots_as_several_lps_per_warp(solver, m, n, dtype):
    sb = _many_pivots(5000, m, n, m + n)
    batch = to_device(sb, dtype)
    got, ref = host(solver.solve(batch, prec="fp32")), host(solver.solve(batch, prec="fp32", kernel=PACK))
    assert ref["iters"].max() > 8 + m * n // (m + n)
    for name in ("status", "iters", "basis", "obj", "x", "y"):
        assert np.array_equal(got[name], ref[name], equal_nan=name == "obj"), name


@pytest.mark.parametrize("prec,rtol", [("fp32", 1e-4), ("fp32_refine", 1e-8)])
@pytest.mark.parametrize("rule", ["lpc", "rpc"])
@pytest.mark.parametrize("m,n,normal", [(40, 33, False), (64, 64, False), (33, 31, True), (60, 50, True), (100, 90, True)])
@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
def test_warm_starts_in_every_mode(solver, prec, rtol, rule, m, n, normal, dtype):
    """Directions that turn slowly, on polytopes whose optimal bases take few pivots and many
    (rows of both signs): each objective starts from the one before under either rule, with
    and without refinement, in batches that fill the GPU (the random rule's route).  Plain FP32:
    some 64 warm pivots and 64 cold ones at 2^-24 times values up to 100, against FP64."""
    r = np.random.default_rng(m + n)
    A = r.normal(0.3, 1, (m, n)) if normal else r.uniform(0.1, 1, (m, n))
    b, count = r.uniform(1, 10, m), 2500
    C = r.uniform(0.1, 1, n)[None] + 1e-5 * np.arange(count)[:, None] * r.normal(size=n)[None]
    args = [torch.tensor(v, device="cuda", dtype=dtype) for v in (A, b, C)]
    got = host(solver.solve_shared(*args, prec=prec, pivot_rule=rule, seed=3))
    ref = host(solver.solve_shared(*[a.double() for a in args], prec="fp64", pivot_rule=rule, seed=3))
    assert np.array_equal(got["status"], ref["status"]) and (ref["status"] == 0).all()
    assert np.all(np.abs(got["obj"] - ref["obj"]) <= rtol * (1 + np.abs(ref["obj"])))
    x, y = got["x"].reshape(count, n), got["y"].reshape(count, m)
    Ad, bd, Cd = (a.double().cpu().numpy() for a in args)
    assert (x @ Ad.T - bd).max() <= rtol * 100 and (Cd - y @ Ad).max() <= rtol * 100 and min(x.min(), y.min()) >= -rtol * 100
    assert got["iters"].mean() < 0.3 * ref["iters"].mean()
    assert solver.sync_error() == 0


# The configurations of 385 to 1,024 rows or columns (eight warps; two and four rows or columns
# per thread), where most of the history lies in the workspace.
@pytest.mark.parametrize("count,m,n", [(12, 385, 40), (12, 512, 30), (12, 513, 40), (12, 40, 1000), (8, 1024, 20),
                                       (6, 530, 600)])
@pytest.mark.parametrize("prec,dtype", [("fp64", torch.float64), ("fp32", torch.float32), ("fp32_refine", torch.float64)])
@pytest.mark.parametrize("many", [False, True])
def test_largest_configurations(solver, count, m, n, prec, dtype, many):
    """LPs of few pivots and (one entry in ten) of many, as above."""
    sb = _many_pivots(count, m, n, m + n, sparse=True) if many else synth.type1(count, m, n, seed=m + n)
    batch = to_device(sb, dtype)
    got, ref = host(solver.solve(batch, prec=prec)), host(solver.solve(batch, prec=prec, kernel=GMEM))
    assert np.array_equal(got["status"], ref["status"])
    if prec == "fp32_refine":
        assert (got["iters"] != ref["iters"]).sum() <= 1       # (an LP solved again, as above)
        ok = ref["status"] == 0
        assert np.all(np.abs(got["obj"][ok] - ref["obj"][ok]) <= 1e-8 * (1 + np.abs(ref["obj"][ok])))
    else:
        for name in ("iters", "basis", "obj", "x", "y"):
            assert np.array_equal(got[name], ref[name], equal_nan=name == "obj"), name
    assert solver.sync_error() == 0


@pytest.mark.parametrize("m,n,prec", [(520, 66, "fp64"), (400, 51, "fp64"), (520, 20, "fp32"), (400, 20, "fp32_refine")])
def test_largest_configurations_under_the_random_rule(solver, m, n, prec):
    """In a batch that fills the GPU: a CTA runs many LPs, one after another."""
    sb = synth.type1(2500, m, n, seed=m)
    batch = to_device(sb)
    got = host(solver.solve(batch, prec=prec, pivot_rule="rpc", seed=5))
    ref = host(solver.solve(batch, prec=prec, pivot_rule="rpc", seed=5, kernel=GMEM))
    assert np.array_equal(got["status"], ref["status"])
    if prec == "fp32_refine":
        assert (got["iters"] != ref["iters"]).sum() <= 50
    else:
        for name in ("iters", "basis", "obj", "x", "y"):
            assert np.array_equal(got[name], ref[name]), name
    assert np.all(np.abs(got["obj"] - ref["obj"]) <= 1e-8 * (1 + np.abs(ref["obj"])))
    assert solver.sync_error() == 0


@pytest.mark.parametrize("count,m,n,prec", [(6000, 33, 31, "fp64"), (4000, 64, 40, "fp64"), (2000, 130, 24, "fp64"),
                                            (6000, 60, 64, "fp32"), (4000, 100, 70, "fp32"), (2500, 140, 30, "fp32")])
def test_nothing_is_left_from_one_lp_to_the_next(solver, count, m, n, prec):
    """Several LPs per CTA, every other one of many pivots."""
    few, many = synth.type1(count, m, n, seed=m), _many_pivots(count, m, n, n)
    sb = synth.pack([(many if k % 2 else few).lp(k) for k in range(count)])
    batch = to_device(sb)
    full = GMEM if prec == "fp64" or max(m, n) > 127 else WARP
    got, ref = host(solver.solve(batch, prec=prec)), host(solver.solve(batch, prec=prec, kernel=full))
    for name in ("status", "iters", "basis", "obj", "x", "y"):
        assert np.array_equal(got[name], ref[name], equal_nan=name == "obj"), name
    assert solver.sync_error() == 0


@pytest.mark.parametrize("call", ["solve", "shared", "bounded", "host"])
@pytest.mark.parametrize("prec", ["fp64", "fp32_refine"])
def test_less_workspace_in_every_call(call, prec):
    """256 bytes less than asked for: the kernels that update the whole tableau, with the same
    statuses and pivots (warm starts of one polytope's objectives: the same optima).  Far
    less: refused."""
    from paper_1609_08114_gb300 import LPBatch, Solver, _lib
    from paper_1609_08114_gb300._lib import LPBError

    class Short(Solver):
        cut, asked = 0, []

        def workspace(self, nbytes):
            self.asked.append(nbytes)
            return torch.empty(max(256, nbytes - self.cut), dtype=torch.uint8, device="cuda")

    s, count, m, n = Short(0), 2500, 90, 80
    sb = synth.type1(count, m, n, seed=8)
    batch = to_device(sb)
    pinned = LPBatch(*(t.cpu().pin_memory() for t in (batch.m, batch.n, batch.a_off, batch.b_off, batch.c_off, batch.A,
                                                      batch.b, batch.c)), batch.max_m, batch.max_n, batch.min_m, batch.min_n)
    run = {"solve": lambda: s.solve(batch, prec=prec), "host": lambda: s.solve_host(pinned, prec=prec, chunk=1000),
           "shared": lambda: s.solve_shared(batch.A[:m * n].view(m, n), batch.b[:m], batch.c.view(count, n), prec=prec),
           "bounded": lambda: s.solve_bounded(batch, torch.zeros_like(batch.c), torch.full_like(batch.c, 0.2), prec=prec)}[call]

    def result():
        r = run()
        torch.cuda.synchronize()
        return {k: getattr(r, k).cpu().numpy().copy() for k in ("status", "iters", "obj")}

    want, kernels = result(), s.stats()["kernels"]
    s.cut = 256
    if call == "bounded" and prec == "fp32_refine":    # its Phase-I slots are the larger ones: nothing to do without
        with pytest.raises(LPBError) as e:
            result()
        assert e.value.code == _lib.ENOMEM
        return
    got = result()
    assert (want["status"] == 0).all() and np.array_equal(got["status"], want["status"])
    if call == "shared" and prec == "fp32_refine":
        assert s.stats()["kernels"] == kernels - 1     # the launch for what the first one leaves
    else:
        assert np.array_equal(got["iters"], want["iters"])
    assert np.all(np.abs(got["obj"] - want["obj"]) <= 1e-8 * (1 + np.abs(want["obj"])))
    s.cut = 1 << 40
    with pytest.raises(LPBError) as e:
        result()
    assert e.value.code == _lib.ENOMEM
    assert s.sync_error() == 0
