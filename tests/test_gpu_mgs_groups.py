"""The grouped Gram-Schmidt step at the edges of its groups, against the oracle's
GMRES, which takes one basis vector at a time (Alg 3.1, GMRES line).

The kernels take the basis in groups of 2, 4 or 8 vectors (one reduction per
group, the triangular form of MGS inside it): step counts on both sides of the
group sizes' multiples reach an empty, a partial and a full last group; grids
of one block (no exchange), two, nine and the default 64 reach the layouts with
and without a spare block for the Givens rotations; the orders leave ragged
last blocks, and rows past the order inside a 16-byte unit.  Bars: those of the
instance tests (fixed steps, 1e-4 in fp32 and 1e-10 in fp64 of the largest
entry); M has one bucket in u_g, so that no product rounds its operand further."""
import numpy as np
import pytest
import torch

import oracle as O
from gpu_helpers import dev, gpu_bucket, host, lib
from paper_2307_03914_gb300 import workloads as W

pytestmark = pytest.mark.gpu

TOL = {"fp32": 1e-4, "fp64": 1e-10}
GRIDS = [(5, 13, 1), (7, 9, 11), (23, 24, 25)]  # n = 65, 693, 13,800


@pytest.fixture(scope="module")
def B():
    return lib()


def _system(B, grid, ug):
    gx, gy, gz = grid
    A = W.convdiff3d(grid) if gz > 1 else W.convdiff2d(gx, gy)
    P = W.pattern_of(A)
    _, b = W.rhs(A)
    muf = O.round_to(O.spai(A, P, 0.3)["mval"], "fp32")
    Mh = B.M_create(B.DeviceCSR(P.n, dev(P.row_ptr), dev(P.col), dev(muf)))
    precs = [ug]
    bk = gpu_bucket(B, Mh, P.nnz, 2.0 ** -37, precs)
    ids = O.bucket_ids(P.row_ptr, muf, 2.0 ** -37, precs)["ids"]
    stored, _, _ = O.bucket_store(P.row_ptr, P.col, muf, ids, precs)
    S = O.System(A, P.row_ptr, P.col, stored, ids, precs)
    r = O.residual_dd(A, O.spmv_prec(P.row_ptr, P.col, muf, "fp32", b), b)
    return A, bk["BM"], S, r


@pytest.mark.parametrize("grid", GRIDS, ids=["65", "693", "13800"])
@pytest.mark.parametrize("ug", ["fp32", "fp64"])
def test_group_edges_match_oracle(B, grid, ug):
    A, BM, S, r = _system(B, grid, ug)
    Ah = B.matrix_create(B.DeviceCSR.from_host(A))
    rd = dev(r)
    for k in (1, 2, 3, 7, 8, 9, 16, 17):
        d_ref, it_ref, res_ref = O.gmres(S, r, ug, ug, 0.0, k)
        for max_blocks in (0, 1, 2, 9):
            if ug == "fp64" and max_blocks == 1 and A.n > 8192:
                continue  # beyond one block's rows: the streaming kernel, as in the next call
            d = torch.empty(A.n, dtype=torch.float64, device="cuda")
            info = B.gmres(Ah, BM, rd, d, ug, ug, B.opts(tau=0.0, kmax=k, max_blocks=max_blocks))
            assert info["gmres_iters"] == [k] and it_ref == k
            err = np.abs(host(d) - d_ref).max() / np.abs(d_ref).max()
            assert err <= TOL[ug], (k, max_blocks, err)


# the one-launch runs: block edges (1,024 and 1,025 rows: one and two row blocks; 32,768:
# the most), two narrow buckets, a mix with fp64 (read from memory), rows of 9 entries
# (the most kept in shared memory) and of 12 (read from memory)
RUNS = [("1024", ["fp32", "fp16"]), ("1025", ["fp32", "fp16"]), ("1025", ["fp64", "fp32", "fp16"]),
        ("9-point", ["fp32"]), ("9-point", ["fp32", "bf16"]), ("rows of 12", ["fp32"]), ("32768", ["fp32", "fp16"])]


@pytest.mark.parametrize("name,precs", RUNS, ids=[f"{n}-{'+'.join(p)}" for n, p in RUNS])
def test_one_launch_runs_match_oracle(B, name, precs):
    A = {"1024": lambda: W.convdiff2d(32, 32), "1025": lambda: W.convdiff2d(25, 41),
         "9-point": lambda: W.convdiff2d_9pt(37), "rows of 12": lambda: W.random_sparse(1500, 11, 1.0, 0.1),
         "32768": lambda: W.convdiff3d(32)}[name]()
    P = W.pattern_of(A)
    eps = 2.0 ** -16
    _, b = W.rhs(A)
    muf = O.round_to(O.spai(A, P, 0.3)["mval"], "fp32")
    Mh = B.M_create(B.DeviceCSR(P.n, dev(P.row_ptr), dev(P.col), dev(muf)))
    bk = gpu_bucket(B, Mh, P.nnz, eps, precs)
    ids = O.bucket_ids(P.row_ptr, muf, eps, precs)["ids"]
    stored, _, _ = O.bucket_store(P.row_ptr, P.col, muf, ids, precs)
    S = O.System(A, P.row_ptr, P.col, stored, ids, precs)
    r = O.residual_dd(A, O.spmv_prec(P.row_ptr, P.col, muf, "fp32", b), b)
    Ah = B.matrix_create(B.DeviceCSR.from_host(A))
    for k in (1, 9, 20):
        d_ref, _, _ = O.gmres(S, r, "fp32", "fp32", 0.0, k)
        d = torch.empty(A.n, dtype=torch.float64, device="cuda")
        n0 = B.launch_count()
        info = B.gmres(Ah, bk["BM"], dev(r), d, "fp32", "fp32", B.opts(tau=0.0, kmax=k))
        assert B.launch_count() - n0 <= 8 and info["gmres_iters"] == [k]  # not three per step
        assert np.abs(host(d) - d_ref).max() <= TOL["fp32"] * np.abs(d_ref).max(), k
    # a run that stops by its tolerance takes the steps the oracle takes
    _, it_ref, _ = O.gmres(S, r, "fp32", "fp32", 1e-3, 200)
    info = B.gmres(Ah, bk["BM"], dev(r), d, "fp32", "fp32", B.opts(tau=1e-3, kmax=200))
    assert abs(info["gmres_iters"][0] - it_ref) <= 1


@pytest.mark.parametrize("ug", ["fp32", "fp64"])
def test_streaming_groups_match_oracle(B, ug):
    """The streaming kernel (one block cannot hold 24,389 rows on chip) over the edges of its groups of four."""
    A, BM, S, r = _system(B, (29, 29, 29), ug)
    assert B.gmres_plan(A.n, ug, 1)["kernel"] == "k_mgs"
    Ah = B.matrix_create(B.DeviceCSR.from_host(A))
    for k in (1, 3, 4, 5, 9):
        d_ref, _, _ = O.gmres(S, r, ug, ug, 0.0, k)
        d = torch.empty(A.n, dtype=torch.float64, device="cuda")
        B.gmres(Ah, BM, dev(r), d, ug, ug, B.opts(tau=0.0, kmax=k, max_blocks=1))
        assert np.abs(host(d) - d_ref).max() <= TOL[ug] * np.abs(d_ref).max(), k
