"""Graphs of more nodes than two 128-byte lines each in L2: blocks of whole
64-column stretches are gathered 256 bytes at a time from plain rows, other widths
and smaller graphs as before.  The width that runs is reported and leaves every
score's bits alone."""
import numpy as np
import pytest

from test_gpu_panels import _queries

pytestmark = pytest.mark.gpu

LINE = (256 << 20) // 128   # nodes


def _graph(ctx, n):
    import torch
    import paper_1807_08692_gb300 as hd
    i = torch.arange(n, device="cuda")
    col = torch.sort(torch.stack([(i + s) % n for s in (1, n - 1, 1000, n - 1000)], 1), 1).values
    return hd.graph_from_csr(ctx, torch.arange(0, 4 * n + 1, 4, device="cuda").int(), col.int().reshape(-1),
                             torch.ones(4 * n, device="cuda"))


@pytest.mark.parametrize("n,widths", [(LINE, {64: 32, 96: 32, 128: 32}), (LINE + 1, {60: 32, 64: 64, 72: 32, 96: 32, 128: 64})])
def test_shape_on_both_sides_of_the_line(gpu_ctx, monkeypatch, n, widths):
    import torch
    import paper_1807_08692_gb300 as hd
    g = _graph(gpu_ctx, n)
    for B, slab in widths.items():
        y = _queries(n, B, np.random.default_rng(B))
        out = []
        for forced in (None, "128"):
            if forced:
                monkeypatch.setenv("HD_SLAB", forced)
            else:
                monkeypatch.delenv("HD_SLAB", raising=False)
            X, it, _, st = hd.query_batch(gpu_ctx, g, None, "paper", *y, 0.9, 1e-4, 60)
            assert np.all(np.array(st) == 0)
            if not forced:
                assert g.tuning(B) == (slab, 1), B
            out.append((X.view(torch.int32), np.array(it)))
        assert np.array_equal(out[0][1], out[1][1]) and bool(torch.equal(out[0][0], out[1][0])), B
    g.close()


SEG = 140 << 20   # bytes of an 8- or 16-column block from which its products take two node ranges


@pytest.mark.parametrize("n,B,segments", [(SEG // 64, 16, 1), (SEG // 64 + 1, 16, 2), (SEG // 64 + 1, 14, 2), (SEG // 64 + 1, 12, 1),
                                          (SEG // 32, 8, 1), (SEG // 32 + 1, 8, 2)])
def test_two_node_ranges(gpu_ctx, monkeypatch, n, B, segments):
    import torch
    import paper_1807_08692_gb300 as hd
    monkeypatch.delenv("HD_SLAB", raising=False)
    g = _graph(gpu_ctx, n)
    y = _queries(n, 20, np.random.default_rng(B))
    k = int(y[0][B])
    X, it, _, st = hd.query_batch(gpu_ctx, g, None, "paper", y[0][:B + 1], y[1][:k], y[2][:k], 0.9, 1e-5, 100)
    assert np.all(np.array(st) == 0) and g.tuning(B)[1] == segments
    # the same columns in a batch of another width, whose sums run in one pass; each residual is below 1e-5 ||y||
    # and L_a >= I, so the two differ by at most 2e-5 ||y||
    W, iw, _, sw = hd.query_batch(gpu_ctx, g, None, "paper", *y, 0.9, 1e-5, 100)
    assert np.all(np.array(sw) == 0) and g.tuning(20)[1] == 1
    ynorm = torch.tensor([float(np.linalg.norm(y[2][y[0][j]:y[0][j + 1]])) for j in range(B)], device="cuda")
    assert bool(((X - W[:, :B]).norm(dim=0) <= 2.1e-5 * ynorm).all())
    assert np.all(np.abs(np.array(it) - np.array(iw)[:B]) <= 1)
    g.close()
