"""k-NN lists when many similarities are equal: runs of identical descriptors,
longer than a list and than a step of the selection, inside one tile, across
tile and segment edges and at the ends of the database, after rows that rank
lower.  Ties go to the smaller id whatever the batch width.  Descriptors are
small integers, so every similarity is exact."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _database(n, d, runs, rng):
    X = rng.integers(-2, 3, (n, d)).astype(np.float32)
    for level, (lo, hi) in enumerate(runs):
        X[lo:hi] = 3.0 + level          # equal to each other, above every random row
    return X


def _reference(X, Q, k, exclude_self):
    S = Q @ X.T
    if exclude_self:
        S[np.arange(S.shape[0]), np.arange(S.shape[0])] = -np.inf
    ids = np.argsort(-S, axis=1, kind="stable")[:, :k]
    return ids.astype(np.int32), np.take_along_axis(S, ids, 1)


# n, runs of identical rows: one tile; a run that starts inside a tile; runs over tile edges, the
# larger value first and last; a run of a whole segment and more; the last rows of a ragged tile
DATABASES = [
    (256, [(128, 256)]), (384, [(130, 250)]), (1000, [(100, 170), (300, 700)]), (1000, [(500, 900), (90, 260)]),
    (5003, [(4000, 5003)]), (5003, [(0, 64), (1500, 3600)]), (40000, [(20000, 20040), (39000, 39900)]),
]


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("nq", [1, 17, 32, 33, 65, 200])   # every tile height of the fp32 kernel and a second block
@pytest.mark.parametrize("n,runs", DATABASES)
def test_ties_go_to_the_smaller_id(gpu_ctx, n, runs, nq, dtype):
    import torch
    import paper_1807_08692_gb300 as hd
    rng = np.random.default_rng(n + nq)
    X = _database(n, 24, runs, rng)
    Q = rng.integers(-2, 3, (nq, 24)).astype(np.float32)
    Q[::2] = 1.0                        # every other query ranks the runs first
    t = torch.bfloat16 if dtype == "bf16" else torch.float32
    Xd, Qd = torch.from_numpy(X).to(t).cuda(), torch.from_numpy(Q).to(t).cuda()
    for k in (1, 5, 10, 33, 50, 64):
        idx, sim = hd.knn(gpu_ctx, Xd, Qd, k)
        ri, rs = _reference(X, Q, k, False)
        assert np.array_equal(idx.cpu().numpy(), ri), k
        assert np.array_equal(sim.cpu().numpy(), rs), k


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("n,runs", [(256, [(128, 256)]), (1000, [(300, 700)]), (5003, [(0, 64), (1500, 3600)])])
def test_ties_without_the_row_itself(gpu_ctx, n, runs, dtype):
    import torch
    import paper_1807_08692_gb300 as hd
    X = _database(n, 24, runs, np.random.default_rng(n))
    t = torch.from_numpy(X).to(torch.bfloat16 if dtype == "bf16" else torch.float32).cuda()
    for k in (1, 10, 50):
        idx, sim = hd.knn(gpu_ctx, t, t, k, exclude_self=True)
        ri, rs = _reference(X, X, k, True)
        assert np.array_equal(idx.cpu().numpy(), ri), k
        assert np.array_equal(sim.cpu().numpy(), rs), k


def test_infinite_and_nan_similarities(gpu_ctx):
    # infinities rank like any value and tie by id; a similarity of -inf or NaN never enters a list
    import torch
    import paper_1807_08692_gb300 as hd
    n = 700
    X = np.random.default_rng(3).integers(-2, 3, (n, 8)).astype(np.float32)
    X[100:260, 0] = np.inf
    X[300:340, 0] = -np.inf
    X[400:410, 0] = np.nan
    Q = np.zeros((3, 8), np.float32)
    Q[:, 0] = 1.0
    Q[1, 1:] = 1.0
    S = Q[:, :1] * X[:, 0] + Q[:, 1:] @ np.nan_to_num(X[:, 1:]).T
    S = np.where(np.isnan(S) | (S == -np.inf), -np.inf, S)
    for k in (7, 50):
        idx, sim = hd.knn(gpu_ctx, torch.from_numpy(X).cuda(), torch.from_numpy(Q).cuda(), k)
        ids = np.argsort(-S, axis=1, kind="stable")[:, :k]
        assert np.array_equal(idx.cpu().numpy(), ids)
        assert np.array_equal(sim.cpu().numpy(), np.take_along_axis(S, ids, 1).astype(np.float32))
    # a database without one finite similarity leaves the places empty
    bad = np.full((40, 8), np.nan, np.float32)
    idx, sim = hd.knn(gpu_ctx, torch.from_numpy(bad).cuda(), torch.from_numpy(Q).cuda(), 5)
    assert np.all(idx.cpu().numpy() == -1) and np.all(sim.cpu().numpy() == -np.inf)
