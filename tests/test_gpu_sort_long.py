"""CSR rows longer than the row sort's buffer: lengths around its multiples, in
ascending, descending, random and nearly sorted order, with repeated columns (which
keep their given order), and the time of such rows."""
import time

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("lengths", [[513, 543, 1023, 1024, 1025, 1537], [2048, 5000, 0, 512], [20011]])
def test_long_rows_are_sorted_stably(gpu_ctx, lengths):
    import paper_1807_08692_gb300 as hd
    rng = np.random.default_rng(sum(lengths))
    n = 30000
    rows = []
    for L in lengths:
        c = np.sort(rng.choice(n, L, replace=False)).astype(np.int32)
        swapped = c.copy()
        swapped[:1], swapped[-1:] = c[-1:], c[:1]
        parts = np.concatenate([c[L // 2:], c[:L // 2]]) if L else c
        rows += [c[::-1].copy(), rng.permutation(c), c, swapped, parts,
                 rng.integers(0, 40, L).astype(np.int32), np.full(L, 7, np.int32), rng.integers(0, n, 5).astype(np.int32)]
    rows += [np.zeros(0, np.int32)] * (n - len(rows))
    rp = np.concatenate([[0], np.cumsum([len(r) for r in rows])]).astype(np.int32)
    col = np.concatenate(rows).astype(np.int32)
    val = np.arange(1, col.size + 1, dtype=np.float32)
    grp, gcol, gval, _ = hd.graph_from_csr(gpu_ctx, rp, col, val, normalized=True).export()
    assert np.array_equal(grp, rp)
    for i in range(8 * len(lengths)):
        order = np.argsort(col[rp[i]:rp[i + 1]], kind="stable")
        assert np.array_equal(gcol[rp[i]:rp[i + 1]], col[rp[i]:rp[i + 1]][order]), i
        assert np.array_equal(gval[rp[i]:rp[i + 1]], val[rp[i]:rp[i + 1]][order]), i


def test_long_rows_take_no_quadratic_time(gpu_ctx):
    # a row of 8,000 entries sorted by one lane's insertions takes seconds
    import torch
    import paper_1807_08692_gb300 as hd
    n, rows, length = 20000, 200, 8000
    rp = torch.clamp(torch.arange(n + 1), max=rows).mul(length).int().cuda()
    col = torch.randint(0, n, (rows * length,), device="cuda").int()
    val = torch.rand(rows * length, device="cuda")
    hd.graph_from_csr(gpu_ctx, rp, col, val).close()
    torch.cuda.synchronize()
    t0 = time.perf_counter()
    hd.graph_from_csr(gpu_ctx, rp, col, val).close()
    torch.cuda.synchronize()
    assert time.perf_counter() - t0 < 0.2


@pytest.mark.parametrize("n", [400, 513, 700])
def test_a_node_that_every_other_picks(gpu_ctx, n):
    # the union graph's row of that node is as long as the graph, on both sides of the sort's limit
    import torch
    import paper_1807_08692_gb300 as hd
    rng = np.random.default_rng(n)
    X = np.zeros((n, 8), np.float32)
    X[:, 1:] = rng.integers(-1, 2, (n, 7))
    X[:, 0] = 1.0
    X[0, 0] = 100.0
    X[0, 1:] = 0.0
    rp, col, val, dinv = hd.build_graph(gpu_ctx, torch.from_numpy(X).cuda(), 3, 1.0).export()
    assert rp[1] - rp[0] == n - 1
    for i in range(n):
        assert np.all(np.diff(col[rp[i]:rp[i + 1]]) > 0), i
