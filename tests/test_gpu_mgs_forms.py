"""Gram-Schmidt forms and orders that the group and instance tests do not reach,
against the oracle's GMRES (Alg 3.1, GMRES line) at a fixed number of steps.

On chip: orders that end inside a 16-byte unit in every instance that copies such
units (fp32 in fours, fp64 in twos; the bulk-copied vectors are rounded up to whole
units, whose rows past the order are zero), with and without a block of its own for
the Givens rotations.  One launch per run: u_g = fp64 with narrow, mixed and uncached products,
u_g = fp32 with two narrow buckets that both hold entries and with fp64 beside fp32,
and more steps than one batch of 32 rotations.  The kernel that ran is told by the
plan and by the number of launches (three per step, or one per run).

Bars: those of the instance tests, 1e-4 (u_g = fp32) and 1e-10 (fp64) of the
largest entry, where products round in u_g only.  A narrow bucket rounds its fp64
operand to fp32: a last bit that differs between the two sides can come out one
fp32 unit apart, so there 2^-24 times the norm bound of ten such entries, 1e-6."""
import numpy as np
import pytest
import torch

import oracle as O
from gpu_helpers import dev, gpu_bucket, host, lib
from paper_2307_03914_gb300 import workloads as W

pytestmark = pytest.mark.gpu

TOL = {"fp32": 1e-4, "fp64": 1e-10}


@pytest.fixture(scope="module")
def B():
    b = lib()
    if torch.cuda.get_device_properties(0).multi_processor_count != 152:
        pytest.skip("instances named for 152 SMs")
    return b


def _system(B, A, precs, eps=2.0 ** -37):
    P = W.pattern_of(A)
    _, b = W.rhs(A)
    muf = O.round_to(O.spai(A, P, 0.3)["mval"], "fp32")
    Mh = B.M_create(B.DeviceCSR(P.n, dev(P.row_ptr), dev(P.col), dev(muf)))
    bk = gpu_bucket(B, Mh, P.nnz, eps, precs)
    ids = O.bucket_ids(P.row_ptr, muf, eps, precs)["ids"]
    assert (np.bincount(ids, minlength=len(precs)) > 0).all()  # no bucket is empty
    stored, _, _ = O.bucket_store(P.row_ptr, P.col, muf, ids, precs)
    S = O.System(A, P.row_ptr, P.col, stored, ids, precs)
    r = O.residual_dd(A, O.spmv_prec(P.row_ptr, P.col, muf, "fp32", b), b)
    return B.matrix_create(B.DeviceCSR.from_host(A)), bk["BM"], S, r


def _check(B, Ah, BM, S, r, ug, k, max_blocks, one_launch, tol):
    d_ref, it_ref, _ = O.gmres(S, r, ug, ug, 0.0, k)
    d = torch.empty(r.size, dtype=torch.float64, device="cuda")
    n0 = B.launch_count()
    info = B.gmres(Ah, BM, dev(r), d, ug, ug, B.opts(tau=0.0, kmax=k, max_blocks=max_blocks))
    launches = B.launch_count() - n0
    assert launches <= 8 if one_launch else launches >= 3 * k + 2
    assert info["gmres_iters"] == [k] and it_ref == k
    err = np.abs(host(d) - d_ref).max() / np.abs(d_ref).max()
    assert err <= tol, (k, err)


# (nx, ny), u_g, max_blocks, rows or pairs per thread, blocks with rows
UNITS = [((129, 131), "fp32", 9, 2, 8),     # n = 16,899, ends three rows into a unit; spare block
         ((569, 58), "fp32", 9, 4, 8),      # 33,002: two
         ((265, 265), "fp32", 9, 12, 8),    # 70,225: one
         ((323, 323), "fp32", 9, 14, 8),    # 104,329: one
         ((346, 347), "fp32", 9, 16, 8),    # 120,062: two
         ((129, 131), "fp32", 2, 12, 2),    # no block to spare
         ((513, 513), "fp32", 0, 4, 64),    # 263,169: reductions polled by bulk copies
         ((115, 113), "fp64", 9, 2, 9),     # 12,995, no block to spare
         ((181, 183), "fp64", 9, 4, 9),     # 33,123
         ((181, 183), "fp64", 20, 2, 19),   # with one
         ((265, 265), "fp64", 20, 4, 19)]


@pytest.mark.parametrize("grid,ug,max_blocks,per_thread,blocks", UNITS,
                         ids=[f"{x * y}-{u}-{m}" for (x, y), u, m, _, _ in UNITS])
def test_orders_that_end_inside_a_unit(B, grid, ug, max_blocks, per_thread, blocks):
    A = W.convdiff2d(*grid)
    plan = B.gmres_plan(A.n, ug, max_blocks)
    assert (plan["per_thread"], plan["blocks"]) == (per_thread, blocks), plan
    Ah, BM, S, r = _system(B, A, [ug])
    for k in (1, 2, 3, 5, 9):
        _check(B, Ah, BM, S, r, ug, k, max_blocks, False, TOL[ug])


def _rows_of_5():
    return W.random_sparse(1700, 4, 2.0, 0.1)


# name, u_g, buckets, eps, bar
RUNS = [("1025", "fp32", ["fp32", "fp16"], 2.0 ** -12, TOL["fp32"]),
        ("1025", "fp32", ["fp64", "fp32"], 2.0 ** -25, TOL["fp32"]),
        ("rows of 5", "fp32", ["fp64", "fp32", "fp16"], 2.0 ** -25, TOL["fp32"]),
        ("1025", "fp64", ["fp32", "fp16"], 2.0 ** -12, 1e-6),
        ("1025", "fp64", ["fp64", "fp32"], 2.0 ** -25, 1e-6),
        ("rows of 5", "fp64", ["fp64", "fp32", "fp16"], 2.0 ** -25, 1e-6),
        ("9-point", "fp64", ["fp64"], 2.0 ** -37, TOL["fp64"]),
        ("rows of 12", "fp64", ["fp64"], 2.0 ** -37, TOL["fp64"])]


@pytest.mark.parametrize("name,ug,precs,eps,tol", RUNS, ids=[f"{n}-{u}-{'+'.join(p)}" for n, u, p, _, _ in RUNS])
def test_one_launch_products(B, name, ug, precs, eps, tol):
    A = {"1025": lambda: W.convdiff2d(25, 41), "rows of 5": _rows_of_5, "9-point": lambda: W.convdiff2d_9pt(37),
         "rows of 12": lambda: W.random_sparse(1500, 11, 1.0, 0.1)}[name]()
    Ah, BM, S, r = _system(B, A, precs, eps)
    for k in (1, 9, 40):
        _check(B, Ah, BM, S, r, ug, k, 0, True, tol)


def test_a_single_fp32_step_is_no_run(B):
    """kmax = 1: in fp32 the three launches of a step, in fp64, and from two steps on, one launch."""
    A = W.convdiff2d(25, 41)
    for ug in ("fp32", "fp64"):
        Ah, BM, S, r = _system(B, A, [ug])
        d = torch.empty(r.size, dtype=torch.float64, device="cuda")
        counts = []
        for k in (1, 2):
            n0 = B.launch_count()
            B.gmres(Ah, BM, dev(r), d, ug, ug, B.opts(tau=0.0, kmax=k))
            counts.append(B.launch_count() - n0)
        assert counts[0] - counts[1] == (2 if ug == "fp32" else 0), (ug, counts)
