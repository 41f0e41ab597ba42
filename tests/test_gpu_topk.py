"""Top-K at the edges of the threshold pass: widths that are and are not
multiples of four, blocks whose element count leaves a remainder, views with
gaps between rows, unaligned bases, ties, infinities, and columns that ask for
nothing.  The order (score descending, id ascending) is unique, so ids and
scores must match exactly."""
import numpy as np
import pytest

from oracle import rank as ORank

pytestmark = pytest.mark.gpu


def _check(ids, sc, x, K):
    for j in range(x.shape[1]):
        k = min(int(K[j]), x.shape[0])
        ref, rs = ORank.topk(x[:, j], k)
        assert np.array_equal(ids[j, :k], ref), j
        assert np.array_equal(sc[j, :k], rs), j
        assert np.all(ids[j, k:] == -1), j


@pytest.mark.parametrize("n,B,K", [(1, 1, 1), (3, 1, 2), (5, 3, 4), (7, 2, 7), (4095, 1, 100), (4097, 5, 10), (9001, 37, 50),
                                   (20011, 64, 100), (33333, 257, 20), (300001, 4, 1000), (1000003, 1, 2048)])
@pytest.mark.parametrize("ties", [False, True])
def test_contiguous_blocks(gpu_ctx, n, B, K, ties):
    import torch
    import paper_1807_08692_gb300 as hd
    rng = np.random.default_rng(n + B)
    x = rng.standard_normal((n, B)).astype(np.float32)
    if ties:
        x = np.round(x * 64) / 64
    if n > 10:
        x[n // 2, 0], x[n // 3, B - 1], x[n // 5, B // 2] = np.inf, -np.inf, -0.0
    Ks = np.full(B, K, np.int32)
    Ks[B // 2:B // 2 + (B > 2)] = 0
    ids, sc = hd.rank(gpu_ctx, torch.from_numpy(x).cuda(), Ks, Kmax=K)
    _check(ids, sc, x, Ks)


@pytest.mark.parametrize("shift", [0, 1, 4])
def test_views(gpu_ctx, shift):
    # rows with gaps (ld > B), and a base `shift` floats into an allocation
    import torch
    import paper_1807_08692_gb300 as hd
    rng = np.random.default_rng(shift)
    n, B, ld = 12345, 20, 24
    flat = rng.standard_normal(n * ld + 8).astype(np.float32)
    t = torch.from_numpy(flat).cuda()
    K = np.full(B, 64, np.int32)
    gaps = t[shift:shift + n * ld].view(n, ld)[:, :B]
    _check(*hd.rank(gpu_ctx, gaps, K), flat[shift:shift + n * ld].reshape(n, ld)[:, :B], K)
    dense = t[shift:shift + n * B].view(n, B)
    _check(*hd.rank(gpu_ctx, dense, K), flat[shift:shift + n * B].reshape(n, B), K)
