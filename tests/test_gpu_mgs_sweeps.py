"""The streamed Gram-Schmidt step with every number of vectors in a sweep, first and
later, against the oracle's GMRES (Alg 3.1, GMRES line).

The kernel takes the basis in groups of four, and a sweep's code is made for the
number of vectors it takes out of the new one and forms products with: steps 1 to 8
and 13 reach each of them.  24,389 rows on one SM, more than it holds; bars: those
of the instance tests."""
import numpy as np
import pytest
import torch

import oracle as O
from gpu_helpers import dev, gpu_bucket, host, lib
from paper_2307_03914_gb300 import workloads as W

pytestmark = pytest.mark.gpu

TOL = {"fp32": 1e-4, "fp64": 1e-10}


@pytest.mark.parametrize("ug", ["fp32", "fp64"])
def test_streamed_sweeps(ug):
    B = lib()
    A = W.convdiff3d(29)
    P = W.pattern_of(A)
    assert B.gmres_plan(A.n, ug, 1)["kernel"] == "k_mgs"
    _, b = W.rhs(A)
    muf = O.round_to(O.spai(A, P, 0.3)["mval"], "fp32")
    Mh = B.M_create(B.DeviceCSR(P.n, dev(P.row_ptr), dev(P.col), dev(muf)))
    bk = gpu_bucket(B, Mh, P.nnz, 2.0 ** -37, [ug])
    ids = O.bucket_ids(P.row_ptr, muf, 2.0 ** -37, [ug])["ids"]
    stored, _, _ = O.bucket_store(P.row_ptr, P.col, muf, ids, [ug])
    S = O.System(A, P.row_ptr, P.col, stored, ids, [ug])
    r = O.residual_dd(A, O.spmv_prec(P.row_ptr, P.col, muf, "fp32", b), b)
    Ah = B.matrix_create(B.DeviceCSR.from_host(A))
    for k in (1, 2, 3, 4, 5, 6, 7, 8, 13):
        d_ref, it_ref, _ = O.gmres(S, r, ug, ug, 0.0, k)
        d = torch.empty(A.n, dtype=torch.float64, device="cuda")
        info = B.gmres(Ah, bk["BM"], dev(r), d, ug, ug, B.opts(tau=0.0, kmax=k, max_blocks=1))
        assert info["gmres_iters"] == [k] and it_ref == k
        assert np.abs(host(d) - d_ref).max() <= TOL[ug] * np.abs(d_ref).max(), k
