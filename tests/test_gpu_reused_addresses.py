"""Captured iterations and the memory of destroyed eigenpairs: a new set of the
same size, with other addresses behind the same one, is solved with its own
arrays (the same bits as in a context that captured nothing before)."""
import ctypes

import numpy as np
import pytest

from _helpers import csr_of, y_arrays

pytestmark = pytest.mark.gpu


def _hold(sizes):
    """Device blocks that take the place of freed ones."""
    rt = ctypes.CDLL("libcudart.so.13")
    out = []
    for s in sizes:
        p = ctypes.c_void_p()
        assert rt.cudaMalloc(ctypes.byref(p), ctypes.c_size_t(s)) == 0
        out.append(p)
    return rt, out


@pytest.mark.parametrize("kind", ["fp8", "f32", "bf16", "sparse"])
def test_new_eigenpairs_of_the_same_size(cfg1_data, kind):
    import paper_1807_08692_gb300 as hd
    args = y_arrays(cfg1_data["yp"], cfg1_data["yi"], cfg1_data["yv"])
    n, r = cfg1_data["U"].shape[0], 40
    rng = np.random.default_rng(11)

    def eigenpairs(ctx, g, s):
        # any orthonormal columns and weights make a valid preconditioner
        U = np.linalg.qr(np.random.default_rng(s).standard_normal((n, r)))[0].astype(np.float32) * (1.0 if s == 0 else 0.5)
        e = hd.eig_from_host(ctx, g, np.linspace(0.95, 0.3, r), U, "f32" if kind == "sparse" else kind)
        if kind == "sparse":
            dense, e = e, e.sparsify(0.5)
            dense.close()
        return e

    def solve(ctx, g, e):
        X, it, rr, st = hd.query_batch(ctx, g, e, "pcg", *args, 0.99, 1e-6, 500)
        return X.cpu().numpy().view(np.uint32), np.array(it)

    ctx, fresh = hd.Context(0), hd.Context(0)
    g = hd.graph_from_csr(ctx, *csr_of(cfg1_data["A"]))
    gf = hd.graph_from_csr(fresh, *csr_of(cfg1_data["A"]))
    ef = eigenpairs(fresh, gf, 1)
    want = solve(fresh, gf, ef)
    held = []
    for attempt in range(4):
        old = eigenpairs(ctx, g, 0)
        for _ in range(3):
            solve(ctx, g, old)
        old.close()
        held.append(_hold([int(s) for s in rng.choice([4 * n, 8 * r, 4 * n * r, 8 * n], 2, replace=False)]))
        new = eigenpairs(ctx, g, 1)
        for _ in range(2):
            got = solve(ctx, g, new)
            assert np.array_equal(got[1], want[1]) and np.array_equal(got[0], want[0]), attempt
        new.close()
    for rt, blocks in held:
        for p in blocks:
            rt.cudaFree(p)
    for c in (ctx, fresh):
        c.close()
