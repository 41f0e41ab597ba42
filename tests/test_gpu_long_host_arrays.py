"""Observations and rankings too long for the pinned staging block are copied from
and to the caller's arrays: the same bits as with device arrays, in calls that mix
long and short ones, and no more pinned memory than the block."""
import numpy as np
import pytest

from test_gpu_panels import _setup

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("count", [2 ** 21, 2 ** 21 + 1, 5 * 10 ** 6])  # up to the block's array limit, one more, several times it
@pytest.mark.parametrize("r", [0, 17])
def test_long_observations(gpu_ctx, count, r):
    import torch
    import paper_1807_08692_gb300 as hd
    n, B = 61000, 128
    g, eig = _setup(gpu_ctx, n, r)
    rng = np.random.default_rng(count)
    per = np.full(B, count // B)
    per[: count % B] += 1
    yp = np.concatenate([[0], np.cumsum(per)]).astype(np.int32)
    yi = np.concatenate([np.sort(rng.choice(n, p, replace=False)) for p in per]).astype(np.int32)
    yv = rng.uniform(0.1, 1.0, count).astype(np.float32)
    out = []
    for y in ((yp, yi, yv), tuple(torch.from_numpy(a).cuda() for a in (yp, yi, yv))):
        X, it, _, st = hd.query_batch(gpu_ctx, g, eig, "pcg" if r else "paper", *y, 0.9, 1e-4, 200)
        assert np.all(np.array(st) == 0)
        out.append((X.cpu().numpy().view(np.uint32), np.array(it)))
    assert np.array_equal(out[0][0], out[1][0]) and np.array_equal(out[0][1], out[1][1])


@pytest.mark.parametrize("B,K", [(1024, 1024), (1025, 1024), (2500, 2048)])  # 8 MiB of results, more, several times as much
def test_long_rankings(gpu_ctx, B, K):
    import torch
    import paper_1807_08692_gb300 as hd
    x = torch.randn((4000, B), device="cuda")
    x[:, 3] = 1.0  # equal scores: the exact path behind the filter
    ids, score = hd.rank(gpu_ctx, x, K)
    want = torch.sort(x, dim=0, descending=True, stable=True)
    assert np.array_equal(np.asarray(score), want.values[:K].T.cpu().numpy())
    assert np.array_equal(np.asarray(ids), want.indices[:K].T.cpu().numpy())


def _resident_kib():
    for line in open("/proc/self/status"):
        if line.startswith("VmRSS"):
            return int(line.split()[1])


def test_a_long_call_leaves_no_long_block():
    import paper_1807_08692_gb300 as hd
    n, B = 61000, 256
    ctx = hd.Context(0)
    g, _ = _setup(ctx, n, 0)
    yp = np.arange(0, n * B + 1, n, dtype=np.int32)
    yi = np.tile(np.arange(n, dtype=np.int32), B)
    yv = np.ones(n * B, np.float32)
    hd.query_batch(ctx, g, None, "paper", yp[:2], yi[:n], yv[:n], 0.5, 1e-2, 5)
    before = _resident_kib()
    hd.query_batch(ctx, g, None, "paper", yp, yi, yv, 0.5, 1e-2, 5)   # 125 MB of observations
    assert _resident_kib() - before < 60 * 1024
    g.close()
    ctx.close()
