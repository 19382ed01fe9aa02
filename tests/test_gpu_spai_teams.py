"""The fixed-pattern SPAI's team instances at the edges of what each holds, against
the oracle's least squares (Alg 2.1 with alpha = 0), with the per-column
perturbation bound of the parity tests.

An instance is chosen by the longest row of the pattern and the most candidates
of a column; its rows are checked per column, and a column whose shadow is larger
is left to the warp-per-column kernel.  The random rows below give blocks on both
sides of each limit: 8 columns and 64 candidates (32 rows, which most shadows
exceed), 12 and 128, 24 and 512 (528 candidates go to the warp-per-column kernel
as a whole), with single rows, ragged last blocks and rank-deficient columns."""
import numpy as np
import pytest
import torch

import oracle as O
from gpu_helpers import gpu_build, lib, spai_tolerance
from paper_2307_03914_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    return lib()


def _case(name):
    if name == "1":
        return W.convdiff2d(1, 1)
    if name == "31":
        return W.convdiff2d(31, 1)
    if name == "9-point":
        return W.convdiff2d_9pt(19)
    k, n = (int(v) for v in name.split("x"))  # k off-diagonal entries per row
    return W.random_sparse(n, k, 1.0, delta=0.1, seed=11 + k)


@pytest.mark.parametrize("name", ["1", "31", "9-point", "4x200", "6x333", "7x257", "8x300", "10x301", "11x129",
                                  "15x400", "21x333", "22x300"])
def test_team_instances_match_oracle(B, name):
    A = _case(name)
    P = W.pattern_of(A)
    g = gpu_build(B, dict(A=A, pattern=P, spai_eps=0.3))
    ref = O.spai(A, P, 0.3)
    assert g["info"]["n_rank_deficient"] == 0 and g["info"]["status"] == 0
    tol = spai_tolerance(ref["kappa"], ref["resid"])
    for k in range(A.n):
        a, b = P.row_ptr[k], P.row_ptr[k + 1]
        e = np.linalg.norm(g["val"][a:b] - ref["mval"][a:b]) / np.linalg.norm(ref["mval"][a:b])
        assert e <= tol[k], (k, e, tol[k])
    assert np.allclose(g["resid"], ref["resid"], rtol=1e-4, atol=1e-6)
    assert g["info"]["n_converged"] == int((g["resid"] <= np.float32(0.3)).sum())
    # the same bits in every run (the columns left over are listed in any order)
    again = gpu_build(B, dict(A=A, pattern=P, spai_eps=0.3))
    assert np.array_equal(again["val"], g["val"]) and np.array_equal(again["resid"], g["resid"])


def test_team_rank_deficient_column(B):
    """Two equal columns in a block: flagged, that row of M zero, its residual one."""
    n = 40
    rows = [[i] for i in range(n)]
    rows[3] = rows[4] = [3, 4]  # rows 3 and 4 of A are equal
    rp = np.cumsum([0] + [len(r) for r in rows]).astype(np.int32)
    A = W.CSR(n, rp, np.concatenate(rows).astype(np.int32), np.ones(rp[-1]))
    A.val[rp[3]:rp[5]] = 2.0
    g = gpu_build(B, dict(A=A, pattern=W.pattern_of(A), spai_eps=0.3))
    assert g["info"]["n_rank_deficient"] == 2 and g["info"]["status"] == B.RANK_DEFICIENT
    assert np.all(g["val"][rp[3]:rp[5]] == 0) and np.all(g["resid"][3:5] == 1)
    keep = np.r_[0:rp[3], rp[5]:rp[-1]]
    assert np.allclose(g["val"][keep], 1.0)
