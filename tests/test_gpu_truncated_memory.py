"""Memory of a truncated call whose shortlists together cover many more ids than
their length (B n large): it grows by a bitmap, the position maps are shared, and
columns on both sides of a share's edge get the bits they get in a smaller call."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_many_columns_on_a_large_graph():
    import torch
    import paper_1807_08692_gb300 as hd
    n, B, s = 200000, 1024, 100
    ctx = hd.Context(0)
    rng = np.random.default_rng(2)
    i = np.arange(n)
    a = np.concatenate([i, (i + 1) % n])
    b = np.concatenate([(i + 1) % n, i])
    order = np.lexsort((b, a))
    g = hd.graph_from_csr(ctx, np.arange(0, 2 * n + 1, 2, dtype=np.int32), b[order].astype(np.int32),
                          rng.uniform(0.1, 1.0, n)[np.minimum(a, b)[order]].astype(np.float32))
    # runs of neighbours, so that the subgraphs have edges
    first = rng.integers(0, n - s, B)
    sl = (first[:, None] + rng.permuted(np.tile(np.arange(s), (B, 1)), axis=1)).astype(np.int32)
    yp = np.arange(B + 1, dtype=np.int32)
    yi = (first + 50).astype(np.int32)
    yv = np.ones(B, np.float32)
    args = (0.9, 1e-5, 200)
    X, it, _, st = hd.temporal_truncated(ctx, g, np.arange(0, B * s + 1, s, dtype=np.int32), sl.reshape(-1), yp, yi, yv, *args)
    X = X.cpu().numpy()
    assert np.all(st == 0) and np.all(X[:, np.arange(B)].max(axis=0) > 0)
    # a map of 4 bytes per id and column was enough before there were bitmaps
    assert ctx.workspace_bytes() <= 4 * B * n
    for lo in range(0, B, 128):
        part = slice(lo, lo + 128)
        x, i2, _, s2 = hd.temporal_truncated(ctx, g, np.arange(0, 128 * s + 1, s, dtype=np.int32), sl[part].reshape(-1),
                                             yp[:129], yi[part], yv[part], *args)
        assert np.array_equal(np.array(i2), np.array(it)[part]) and np.array_equal(np.array(s2), np.array(st)[part])
        assert np.array_equal(x.cpu().numpy().view(np.uint32), X[:, part].copy().view(np.uint32)), lo
    g.close()
    ctx.close()
