"""The counters of the fixed-pattern SPAI against the per-column results they sum up.

A block of the narrow team instances solves 32 columns by eight warps that share
no barrier, and adds its counts in shared memory: every count has to arrive
whichever warp is done first.  Empty and one-entry rows of the pattern, whose
warps have next to nothing to do, stand beside full ones and beside pairs of
equal rows (rank deficient), in whole blocks of each kind and mixed within a
warp, over repeated builds."""
import numpy as np
import pytest

from gpu_helpers import gpu_build, lib
from paper_2307_03914_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _matrices(n, width, run):
    """A band of `width` entries per row whose rows come in equal pairs at every 16th row, and a
    pattern whose rows go empty, single, full in runs of `run` rows."""
    half = width // 2
    rows, vals = [], []
    rng = np.random.default_rng(7 * width + run)
    for i in range(n):
        c = np.unique(np.clip(np.arange(i - half, i + half + 1), 0, n - 1))
        v = rng.uniform(0.1, 1.0, c.size)
        v[c == i] += width
        if i % 16 == 1:  # equal to the row before
            c, v = rows[i - 1], vals[i - 1]
        rows.append(c)
        vals.append(v)
    rp = np.cumsum([0] + [r.size for r in rows]).astype(np.int32)
    A = W.CSR(n, rp, np.concatenate(rows).astype(np.int32), np.concatenate(vals))
    kind = (np.arange(n) // run) % 3
    prow = [np.array([], int) if t == 0 else np.array([i]) if t == 1 else
            np.unique(np.clip(np.arange(i - half, i + half + 1), 0, n - 1)) for i, t in enumerate(kind)]
    prp = np.cumsum([0] + [r.size for r in prow]).astype(np.int32)
    P = W.CSR(n, prp, np.concatenate(prow).astype(np.int32), np.ones(prp[-1]))
    return A, P


@pytest.mark.parametrize("width", [5, 7, 11])
@pytest.mark.parametrize("run", [1, 4, 32])
def test_counts_match_the_columns(width, run):
    B = lib()
    A, P = _matrices(8500, width, run)
    eps = 0.2
    for rep in range(8):
        g = gpu_build(B, dict(A=A, pattern=P, spai_eps=eps))
        rp = P.row_ptr
        zero = np.array([rp[k + 1] > rp[k] and not g["val"][rp[k]:rp[k + 1]].any() for k in range(P.n)])
        info = g["info"]
        assert zero.any() and info["n_rank_deficient"] == int((zero & (g["resid"] == 1)).sum()), rep
        assert info["n_converged"] == int((g["resid"] <= np.float32(eps)).sum()), rep
        assert info["max_resid"] == g["resid"].max(), rep
        assert info["status"] == B.RANK_DEFICIENT, rep
