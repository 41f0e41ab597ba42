"""k-NN lists at the edges of the search's tiles, segments and lists.  The
descriptors are small integers, so every similarity is exact in fp32 in any
order of summation and ties are frequent: the lists must equal the reference's
(similarity descending, then id ascending) entry for entry."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

CASES = [
    # n, nq, d, k: one tile, its neighbours, ragged tails, k at the edges of a warp's registers, n < k,
    # one query block against many segments, more query blocks than the GPU has SMs
    (1, 1, 8, 1), (5, 3, 8, 9), (255, 1, 64, 10), (256, 128, 64, 32), (257, 129, 72, 33), (1000, 64, 200, 64),
    (4097, 7, 136, 50), (60000, 65, 64, 10), (30000, 300, 24, 50), (3000, 20001, 16, 31),
]


def _reference(X, Q, k, exclude_self):
    idx = np.full((Q.shape[0], k), -1, np.int32)
    sim = np.full((Q.shape[0], k), -np.inf, np.float32)
    for s0 in range(0, Q.shape[0], 1024):
        S = Q[s0:s0 + 1024] @ X.T
        if exclude_self:
            S[np.arange(S.shape[0]), np.arange(s0, s0 + S.shape[0])] = -np.inf
        m = min(k, X.shape[0] - int(exclude_self))
        # exact integers: one sortable value per entry, larger similarity first, then smaller id
        key = S.astype(np.float64) * X.shape[0] - np.arange(X.shape[0])
        top = np.argsort(-key, axis=1)[:, :m]
        idx[s0:s0 + 1024, :m] = top
        sim[s0:s0 + 1024, :m] = np.take_along_axis(S, top, 1)
    return idx, sim


@pytest.mark.parametrize("dtype", ["bf16", "f32"])
@pytest.mark.parametrize("n,nq,d,k", CASES)
def test_lists_equal_the_exact_order(gpu_ctx, n, nq, d, k, dtype):
    import torch
    import paper_1807_08692_gb300 as hd
    rng = np.random.default_rng(n + nq)
    X = rng.integers(-2, 3, (n, d)).astype(np.float32)
    Q = rng.integers(-2, 3, (nq, d)).astype(np.float32)
    t = torch.bfloat16 if dtype == "bf16" else torch.float32
    idx, sim = hd.knn(gpu_ctx, torch.from_numpy(X).to(t).cuda(), torch.from_numpy(Q).to(t).cuda(), k)
    ri, rs = _reference(X, Q, k, False)
    assert np.array_equal(idx.cpu().numpy(), ri)
    assert np.array_equal(sim.cpu().numpy(), rs)


@pytest.mark.parametrize("dtype", ["bf16", "f32"])
@pytest.mark.parametrize("n,d,k", [(2, 8, 1), (129, 64, 50), (2000, 40, 30), (20100, 16, 64)])
def test_self_is_excluded(gpu_ctx, n, d, k, dtype):
    import torch
    import paper_1807_08692_gb300 as hd
    X = np.random.default_rng(n).integers(-2, 3, (n, d)).astype(np.float32)
    t = torch.from_numpy(X).to(torch.bfloat16 if dtype == "bf16" else torch.float32).cuda()
    idx, sim = hd.knn(gpu_ctx, t, t, k, exclude_self=True)
    ri, rs = _reference(X, X, k, True)
    assert np.array_equal(idx.cpu().numpy(), ri)
    assert np.array_equal(sim.cpu().numpy(), rs)
