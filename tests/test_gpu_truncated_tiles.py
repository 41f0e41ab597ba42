"""Truncated systems at the edges of their streamed products: rows without
entries (first, last, in between), rows longer than a tile, one row, one column,
more columns than a block's share, columns that stop early and shortlists of
different lengths, against a dense fp64 solve of each subsystem."""
import numpy as np
import pytest
import scipy.sparse as sp

from _helpers import csr_of, rel_l2_cols
from oracle import truncated as T

pytestmark = pytest.mark.gpu


def _graph(n, degree, hubs, rng):
    i = rng.integers(0, n, n * degree)
    j = rng.integers(0, n, n * degree)
    for h in range(hubs):  # a node linked to everything
        i = np.concatenate([i, np.full(n, h)])
        j = np.concatenate([j, np.arange(n)])
    keep = (i != j) & (i % 7 != 3) & (j % 7 != 3)  # every seventh node has no edge
    A = sp.csr_matrix((rng.uniform(0.05, 1.0, keep.sum()), (i[keep], j[keep])), shape=(n, n))
    return A.maximum(A.T).tocsr()


@pytest.mark.parametrize("n,degree,hubs,sizes", [
    (50, 2, 0, [1, 7, 50]), (3000, 3, 1, [3000]), (6000, 2, 2, [6000, 1, 2500, 5999, 3]),
    (1500, 6, 0, [300 + 40 * k for k in range(30)]),
])
def test_against_the_subsystem_solve(gpu_ctx, n, degree, hubs, sizes):
    import paper_1807_08692_gb300 as hd
    rng = np.random.default_rng(n + len(sizes))
    A = _graph(n, degree, hubs, rng)
    g = hd.graph_from_csr(gpu_ctx, *csr_of(A))
    B = len(sizes)
    sls = [rng.permutation(n)[:s].astype(np.int32) for s in sizes]
    slp = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int32)
    # observations on the shortlist; the tolerances make the columns stop at different iterations
    yi = np.concatenate([np.sort(s[:3]) for s in sls]).astype(np.int32)
    yp = np.concatenate([[0], np.cumsum([min(3, s) for s in sizes])]).astype(np.int32)
    yv = rng.uniform(0.1, 1.0, yi.size).astype(np.float32)
    tol = np.where(np.arange(B) % 5 == 4, 1e-2, 1e-6).astype(np.float32)
    X, it, rr, st = hd.temporal_truncated(gpu_ctx, g, slp, np.concatenate(sls), yp, yi, yv, 0.9, tol, 500)
    X = X.cpu().numpy().astype(np.float64)
    for j in range(B):
        y = np.zeros(n)
        y[yi[yp[j]:yp[j + 1]]] = yv[yp[j]:yp[j + 1]]
        ref, _ = T.temporal_truncated(A, sls[j], y, 0.9, 1e-12, 5000)
        # a residual of tol ||y|| is an error of at most tol ||y|| <= tol ||x|| / (1 - alpha) (L_a >= I, x >= (1 - a) y)
        bound = 10 * tol[j] + 1e-5
        assert rel_l2_cols(X[:sizes[j], j:j + 1], ref[:, None]).max() <= bound, j
        assert np.all(X[sizes[j]:, j] == 0.0)
