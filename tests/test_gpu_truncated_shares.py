"""Truncated systems whose shortlists differ much in length: empty ones first, last
and in between, one that holds nearly all rows, more columns than one scan takes,
columns that stop at different iterations.  Each column gets the bits it gets in a
call of its own, and a long shortlist is not held up by short ones beside it."""
import time

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _graph(ctx, n, degree):
    import torch
    import paper_1807_08692_gb300 as hd
    g = torch.Generator(device="cuda")
    g.manual_seed(n)
    near = torch.arange(n, device="cuda")[:, None] + torch.randint(1, 60, (n, degree), generator=g, device="cuda")
    a = torch.arange(n, device="cuda").repeat_interleave(degree)
    b = (near % n).reshape(-1)
    key = torch.unique(torch.cat([a * n + b, b * n + a]))
    row, col = key // n, key % n
    rp = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    rp[1:] = torch.cumsum(torch.bincount(row, minlength=n), 0)
    # symmetric weights from the pair's ids
    lo, hi = torch.minimum(row, col), torch.maximum(row, col)
    return hd.graph_from_csr(ctx, rp.int(), col.int(), ((lo * 31 + hi * 17) % 97 + 3).float() / 100)


def _inputs(n, sizes, rng):
    """Per shortlist a run of neighbouring ids in random order, and one observation in it."""
    sls, obs = [], []
    for s in sizes:
        first = int(rng.integers(0, n - s + 1))
        sls.append(rng.permutation(np.arange(first, first + s)).astype(np.int32))
        obs.append(int(sls[-1][0]) if s else 0)
    return np.concatenate([[0], np.cumsum(sizes)]).astype(np.int32), sls, np.array(obs, np.int32)


@pytest.mark.parametrize("n,sizes", [
    (3000, [0, 3000, 0, 1, 0]), (5000, [1] * 40 + [5000]), (5000, [4000] + [0] * 30 + [7, 0, 900]),
    (20000, [20000, 33, 64, 1023, 1025]), (4000, [(37 * j) % 90 for j in range(1100)]),
])
def test_columns_equal_their_own_calls(gpu_ctx, n, sizes):
    import paper_1807_08692_gb300 as hd
    rng = np.random.default_rng(n + len(sizes))
    g = _graph(gpu_ctx, n, 4)
    B = len(sizes)
    ptr, sls, obs = _inputs(n, sizes, rng)
    yp, yv = np.arange(B + 1, dtype=np.int32), np.ones(B, np.float32)
    tol = np.where(np.arange(B) // 4 % 3 == 1, 1e-1, 1e-5).astype(np.float32)  # quads that stop early
    X, it, _, st = hd.temporal_truncated(gpu_ctx, g, ptr, np.concatenate(sls), yp, obs, yv, 0.9, tol, 200)
    X, it, st = X.cpu().numpy(), np.array(it), np.array(st)
    smax = max(sizes)
    for j in (range(B) if B < 100 else list(range(0, B, 53)) + [1022, 1023, 1024, 1099]):
        assert np.all(X[sizes[j]:, j] == 0.0), j
        if sizes[j] == 0:
            continue
        # (beside an empty list of the full length, the reductions take the same chunks of rows)
        pair = np.array([0, sizes[j], sizes[j] + smax], np.int32)
        fill = rng.permutation(n)[:smax].astype(np.int32)
        x, i1, _, s1 = hd.temporal_truncated(gpu_ctx, g, pair, np.concatenate([sls[j], fill]), np.array([0, 1, 1], np.int32),
                                             obs[j:j + 1], np.ones(1, np.float32), 0.9, tol[j], 200)
        assert it[j] == i1[0] and st[j] == s1[0], j
        assert np.array_equal(x.cpu().numpy()[:, 0].copy().view(np.uint32), X[:, j].copy().view(np.uint32)), j


def test_a_long_shortlist_among_short_ones(gpu_ctx):
    import torch
    import paper_1807_08692_gb300 as hd
    n = 400000
    g = _graph(gpu_ctx, n, 16)
    rng = np.random.default_rng(1)

    def seconds(sizes):
        ptr, sls, obs = _inputs(n, sizes, rng)
        B = len(sizes)
        idx, X = torch.from_numpy(np.concatenate(sls)).cuda(), torch.empty((max(sizes), B), device="cuda")
        best = 1e9
        for _ in range(6):
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            hd.temporal_truncated(gpu_ctx, g, ptr, idx, np.arange(B + 1, dtype=np.int32), obs, np.ones(B, np.float32),
                                  0.99, 1e-12, 40, X=X)
            torch.cuda.synchronize()
            best = min(best, time.perf_counter() - t0)
        return best

    # the products of the long one take all of the GPU either way; the vectors are four times as wide
    assert seconds([300000] + [500] * 15) < 2.5 * seconds([300000])


def test_short_shortlists_run_side_by_side(gpu_ctx):
    import torch
    import paper_1807_08692_gb300 as hd
    n = 20000
    g = _graph(gpu_ctx, n, 16)
    rng = np.random.default_rng(4)

    def seconds(B):
        ptr, sls, obs = _inputs(n, [100] * B, rng)
        idx, X = torch.from_numpy(np.concatenate(sls)).cuda(), torch.empty((100, B), device="cuda")
        best = 1e9
        for _ in range(12):
            torch.cuda.synchronize()
            t0 = time.perf_counter()
            hd.temporal_truncated(gpu_ctx, g, ptr, idx, np.arange(B + 1, dtype=np.int32), obs, np.ones(B, np.float32),
                                  0.99, 1e-12, 100, X=X)
            torch.cuda.synchronize()
            best = min(best, time.perf_counter() - t0)
        return best

    # sixteen short chains of loads take the time of one, not of sixteen in a block
    assert seconds(16) < 1.3 * seconds(1)
