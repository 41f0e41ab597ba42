"""Contexts on several threads at once, sharing one graph and one set of
eigenpairs: every thread's first and later solves, rankings and truncated solves
give the bits of the same calls made alone."""
import threading

import numpy as np
import pytest

from _helpers import csr_of

pytestmark = pytest.mark.gpu


def test_contexts_on_threads_share_a_graph(gpu_ctx, cfg1_data):
    import torch
    import paper_1807_08692_gb300 as hd
    n = cfg1_data["U"].shape[0]
    g = hd.graph_from_csr(gpu_ctx, *csr_of(cfg1_data["A"]))
    eig = hd.eig_from_host(gpu_ctx, g, cfg1_data["lam"][:30], cfg1_data["U"][:, :30], "bf16")
    widths = list(range(1, 65, 3))

    def calls(ctx, order):
        out = {}
        for B in order:
            rng = np.random.default_rng(B)
            y = (np.arange(0, 3 * B + 1, 3, dtype=np.int32),
                 np.concatenate([np.sort(rng.choice(n, 3, replace=False)) for _ in range(B)]).astype(np.int32),
                 rng.uniform(0.1, 1.0, 3 * B).astype(np.float32))
            X, it, _, st = hd.query_batch(ctx, g, eig, "pcg", *y, 0.99, 1e-5, 500)
            ids, _ = hd.rank(ctx, X, 20)
            sl = np.concatenate([rng.permutation(n)[:300] for _ in range(B)]).astype(np.int32)
            T, i2, _, _ = hd.temporal_truncated(ctx, g, np.arange(0, 300 * B + 1, 300, dtype=np.int32), sl, *y, 0.9, 1e-4, 100)
            out[B] = [X.cpu().numpy().view(np.uint32), np.array(it), np.asarray(ids), T.cpu().numpy().view(np.uint32), np.array(i2)]
        return out

    results, errors = {}, []
    start = threading.Barrier(6)

    def work(k):
        try:
            stream = torch.cuda.Stream()
            order = np.random.default_rng(k).permutation(widths).tolist()
            with torch.cuda.stream(stream):
                ctx = hd.Context(0, stream=stream)
                start.wait()
                results[k] = calls(ctx, order)
                ctx.close()
        except Exception as e:  # reported by the main thread
            errors.append((k, e))
            start.abort()

    threads = [threading.Thread(target=work, args=(k,)) for k in range(6)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
    want = calls(gpu_ctx, widths)
    for k, got in results.items():
        for B in widths:
            for a, b in zip(got[B], want[B]):
                assert np.array_equal(a, b), (k, B)
