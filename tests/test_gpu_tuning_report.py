"""The reported SpMM shape is the one that runs: panels of 32 columns where a wide
or ragged block is kept in them, the slab of plain rows elsewhere (a forced width,
narrow or small blocks)."""
import numpy as np
import pytest

from test_gpu_panels import _queries, _setup

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,B,panels,rows", [(61000, 72, 32, 8), (61000, 48, 48, 16), (61000, 64, 64, 64),
                                             (262144, 256, 32, 128)])
def test_reported_width(gpu_ctx, monkeypatch, n, B, panels, rows):
    import paper_1807_08692_gb300 as hd
    g, _ = _setup(gpu_ctx, n, 0)
    y = _queries(n, B, np.random.default_rng(1))
    for slab, want in ((None, panels), ("128", rows)):
        if slab:
            monkeypatch.setenv("HD_SLAB", slab)
        else:
            monkeypatch.delenv("HD_SLAB", raising=False)
        hd.query_batch(gpu_ctx, g, None, "paper", *y, 0.9, 1e-2, 20)
        assert g.tuning(B) == (want, 1)
