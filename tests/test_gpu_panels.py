"""Directions kept in panels of a 128-byte line against the plain row layout (a
forced slab width takes it): the same bits, at widths whose last panel is a whole
one, joined, or one column quad, with and without eigenpairs and fp16 gathers."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _setup(ctx, n, r):
    import paper_1807_08692_gb300 as hd
    rng = np.random.default_rng(n)
    i = np.arange(n)
    src = np.concatenate([i, i, rng.integers(0, n, n)])
    dst = np.concatenate([(i + 1) % n, (i + 1000) % n, rng.integers(0, n, n)])
    keep = src != dst
    a, b = np.concatenate([src[keep], dst[keep]]), np.concatenate([dst[keep], src[keep]])
    order = np.lexsort((b, a))
    rp = np.concatenate([[0], np.cumsum(np.bincount(a, minlength=n))]).astype(np.int32)
    w = np.full(a.size, 1.0, np.float32)
    g = hd.graph_from_csr(ctx, rp, b[order].astype(np.int32), w)
    if r == 0:
        return g, None
    # any orthonormal columns and weights make a valid preconditioner
    U = np.linalg.qr(rng.standard_normal((n, r)))[0].astype(np.float32)
    return g, hd.eig_from_host(ctx, g, np.linspace(0.95, 0.3, r), U, "bf16")


def _queries(n, B, rng):
    k = 3
    idx = np.concatenate([np.sort(rng.choice(n, k, replace=False)) for _ in range(B)]).astype(np.int32)
    val = rng.uniform(0.1, 1.0, B * k).astype(np.float32)
    return np.arange(0, B * k + 1, k, dtype=np.int32), idx, val


@pytest.mark.parametrize("n,widths,r", [
    (61000, (70, 88, 148), 0),          # 16 MB and more: narrow last panels joined
    (61000, (72, 104), 17),
    (530000, (33, 52, 72, 104), 0),     # larger than L2: any last panel alone
    (262144, (256, 100), 8),            # whole panels from 256 MB on
])
def test_panels_equal_rows(gpu_ctx, monkeypatch, n, widths, r):
    import paper_1807_08692_gb300 as hd
    g, eig = _setup(gpu_ctx, n, r)
    rng = np.random.default_rng(7)
    for B in widths:
        y = _queries(n, B, rng)
        y[2][:6] = 0.0  # two columns without an observation
        tol = np.where(np.arange(B) % 3 == 1, 1e-2, 1e-5).astype(np.float32)
        out = []
        for slab in (None, "128"):
            if slab:
                monkeypatch.setenv("HD_SLAB", slab)
            else:
                monkeypatch.delenv("HD_SLAB", raising=False)
            X, it, rr, st = hd.query_batch(gpu_ctx, g, eig, "pcg" if r else "paper", *y, 0.95, tol, 300)
            out.append((X.cpu().numpy(), np.array(it), np.array(st)))
        assert np.array_equal(out[0][1], out[1][1]) and np.array_equal(out[0][2], out[1][2]), B
        assert np.array_equal(out[0][0].view(np.uint32), out[1][0].view(np.uint32)), B


def test_server_lanes_with_panels(gpu_ctx):
    # a request alone in the narrow lane (rows) and in a crowd (a lane of 72 columns in panels)
    import paper_1807_08692_gb300 as hd
    n, slots = 61000, 72
    g, eig = _setup(gpu_ctx, n, 17)
    ptr, idx, val = _queries(n, slots, np.random.default_rng(3))
    req = [(idx[ptr[j]:ptr[j + 1]], val[ptr[j]:ptr[j + 1]]) for j in range(slots)]
    srv = hd.Server(gpu_ctx, g, eig, "pcg", 0.95, max_slots=slots, max_iter=300, Kmax=50)
    got = []
    for batch in ([req[5]], req, req[:40] + [req[5]]):
        tickets = [srv.submit(i, v, 1e-5, 50) for i, v in batch]
        while srv.step(1):
            pass
        got.append([srv.poll(t, 50) for t in tickets])
    srv.close()
    a = got[0][0]
    for m in (got[1][5], got[2][40], got[2][5]):
        assert np.array_equal(a[0], m[0]) and np.array_equal(a[1].view(np.uint32), m[1].view(np.uint32))
        assert a[2]["iters"] == m[2]["iters"] and m[2]["status"] == 0
