"""The column reductions stream their blocks at about the rate of a device copy of
the same bytes, at widths and sizes on both sides of the rule that picks their form."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _copy_us_per_gb(torch):
    a = torch.empty(1 << 28, dtype=torch.float32, device="cuda")
    b = torch.empty_like(a)
    best = 1e9
    for _ in range(8):
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        b.copy_(a)
        e1.record()
        torch.cuda.synchronize()
        best = min(best, e0.elapsed_time(e1))
    return best * 1e3 / (2 * a.numel() * 4 / 1e9)


def _times_us(hd, n, B):
    import torch
    ctx = hd.Context(0)
    ctx.profile(True)
    i = torch.arange(n, device="cuda")
    col = torch.sort(torch.stack([(i + s) % n for s in (1, n - 1, 1000, n - 1000)], 1), 1).values
    g = hd.graph_from_csr(ctx, torch.arange(0, 4 * n + 1, 4, device="cuda").int(), col.int().reshape(-1),
                          torch.ones(4 * n, device="cuda"))
    y = (np.arange(B + 1, dtype=np.int32), np.random.default_rng(0).integers(0, n, B).astype(np.int32), np.ones(B, np.float32))
    X = torch.empty((n, B), device="cuda")
    best = {}
    for _ in range(5):
        for f in ("dot", "update"):
            ctx.profile_read(f)
        hd.query_batch(ctx, g, None, "paper", *y, 0.99, 1e-9, 6, X=X)
        for f in ("dot", "update"):
            c, ms = ctx.profile_read(f)
            best[f] = min(best.get(f, 1e9), ms / c * 1e3)
    g.close()
    ctx.close()
    return best


@pytest.mark.parametrize("n,B", [(1000000, 64)])
def test_streams_at_the_copy_rate(n, B):
    import torch
    import paper_1807_08692_gb300 as hd
    rate = _copy_us_per_gb(torch)
    t = _times_us(hd, n, B)
    gb = n * B * 4 / 1e9
    # two blocks read; four read and two written
    assert t["dot"] < 1.33 * rate * 2 * gb and t["update"] < 1.05 * rate * 6 * gb, (t, rate)


@pytest.mark.parametrize("n,B", [(300000, 128), (1000000, 36), (500000, 100)])
def test_half_full_grids_are_not_staged(n, B):
    # sizes whose thread form has 700 to 1,000 threads per SM: staged they ran at half this rate
    import torch
    import paper_1807_08692_gb300 as hd
    rate = _copy_us_per_gb(torch)
    t = _times_us(hd, n, B)
    gb = n * B * 4 / 1e9
    assert t["dot"] < 1.8 * rate * 2 * gb and t["update"] < 1.2 * rate * 6 * gb, (t, rate)
