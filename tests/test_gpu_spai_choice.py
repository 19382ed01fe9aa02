"""Which form of the fixed-pattern SPAI solves which columns.

A narrow team holds 32 rows.  Where a sample of the columns (above 8,192 of them)
says that most shadows are taller, the whole build goes to one launch of another form; where few
are, the team leaves those to one more launch.  No column is solved by both.
Against the oracle's least squares with the bound of the parity tests, and by the
number of launches against a build in half, which always has one solving launch."""
import numpy as np
import pytest

import oracle as O
from gpu_helpers import gpu_build, lib, spai_tolerance
from paper_2307_03914_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    return lib()


def _launches(B, A, u_f):
    Ad, Pd = B.DeviceCSR.from_host(A), B.DeviceCSR.from_host(A, with_values=False)
    n0 = B.launch_count()
    M, _ = B.bspai_build(Ad, Pd, 0.3, u_f=u_f)
    return B.launch_count() - n0


def _with_scattered_rows(A0, part, k):
    """The first `part` of the rows replaced by the diagonal and k - 1 random columns."""
    rng = np.random.default_rng(17)
    rows = [A0.col[A0.row_ptr[i]:A0.row_ptr[i + 1]] for i in range(A0.n)]
    vals = [A0.val[A0.row_ptr[i]:A0.row_ptr[i + 1]] for i in range(A0.n)]
    for i in range(int(A0.n * part)):
        rows[i] = np.unique(np.r_[rng.integers(0, A0.n, k - 1), i])
        vals[i] = np.where(rows[i] == i, 2.0 * k, rng.uniform(-1.0, 1.0, rows[i].size))
    rp = np.cumsum([0] + [r.size for r in rows]).astype(np.int32)
    return W.CSR(A0.n, rp, np.concatenate(rows).astype(np.int32), np.concatenate(vals))


def _band(n, w):
    cols = np.sort((np.arange(n)[:, None] + np.arange(-(w // 2), w - w // 2)) % n, axis=1)
    vals = np.random.default_rng(5).uniform(-1.0, 1.0, cols.shape)
    vals[cols == np.arange(n)[:, None]] = 1.5 * w
    return W.CSR(n, (np.arange(n + 1) * w).astype(np.int32), cols.reshape(-1).astype(np.int32), vals.reshape(-1))


def _match(B, A):
    P = W.pattern_of(A)
    g = gpu_build(B, dict(A=A, pattern=P, spai_eps=0.3))
    ref = O.spai(A, P, 0.3)
    tol = spai_tolerance(ref["kappa"], ref["resid"])
    for k in range(A.n):
        a, b = P.row_ptr[k], P.row_ptr[k + 1]
        e = np.linalg.norm(g["val"][a:b] - ref["mval"][a:b]) / np.linalg.norm(ref["mval"][a:b])
        assert e <= tol[k], (k, e, tol[k])
    assert np.allclose(g["resid"], ref["resid"], rtol=1e-4, atol=1e-6)
    assert g["info"]["n_converged"] == int((g["resid"] <= np.float32(0.3)).sum())


# |J| scattered entries per row: every shadow taller than a narrow team (7, 9, 11), no instance
# that holds the candidates and pays (13), the wide team (15: 225 candidates)
@pytest.mark.parametrize("k", [6, 8, 10, 12, 14])
@pytest.mark.parametrize("n", [1500, 9000])
def test_scattered_columns_are_solved_once(B, n, k):
    A = W.random_sparse(n, k, 1.0, delta=0.1, seed=3 + k)
    assert _launches(B, A, "fp32") == _launches(B, A, "fp16")


@pytest.mark.parametrize("name,part", [("7-point", 0.0), ("9-point", 0.0), ("7-point", 0.25), ("9-point", 0.25), ("7-point", 0.75), ("9-point", 0.75)])
def test_columns_left_by_a_team(B, name, part):
    A0, k = (W.convdiff3d((19, 21, 22)), 7) if name == "7-point" else (W.convdiff2d_9pt(93), 9)
    A = _with_scattered_rows(A0, part, k)
    assert _launches(B, A, "fp32") - _launches(B, A, "fp16") == (1 if 0 < part < 0.5 else 0)
    _match(B, A)


@pytest.mark.parametrize("w", [12, 13, 14, 16, 17])
def test_bands(B, w):
    """Low shadows of 144 to 289 candidates: a warp per column up to 256, the wide team above."""
    A = _band(8600, w)
    assert _launches(B, A, "fp32") == _launches(B, A, "fp16")
    _match(B, A)
