"""Walks of layouts far beyond L2 (loads that are fetched by 64 bytes) against
the same walks of a statistics launch, which reads them the ordinary way."""
import numpy as np
import pytest

from paper_1903_11749_gb300 import ppr

pytestmark = pytest.mark.gpu


def test_far_layout_walks_the_same():
    import torch

    l2 = torch.cuda.get_device_properties(0).L2_cache_size
    d = 24
    n = int(16.5 * l2 / 16) // d  # alias slots (16 bytes an edge) just above 16 times the L2, guide slots well above
    g = torch.Generator(device="cuda").manual_seed(3)
    # rows of 1 to 47 edges, a few without any (they restart); weights 1 .. 1,000
    deg = torch.randint(1, 2 * d, (n,), generator=g, device="cuda")
    deg[::97] = 0
    rp = torch.zeros(n + 1, dtype=torch.int64, device="cuda")
    rp[1:] = torch.cumsum(deg, 0)
    m = int(rp[-1])
    col = torch.randint(0, n, (m,), generator=g, device="cuda", dtype=torch.int32)
    w = torch.randint(1, 1001, (m,), generator=g, device="cuda", dtype=torch.int32)
    ctx = ppr.Context(0)
    G = ctx.load_graph(n, rp, col, w, m=m)
    for kw in (dict(), dict(sampler=1), dict(segments=True)):
        far = G.run(alpha=0.15, R=40, seed=9, topk=8, src_begin=n - 3000, src_end=n, **kw)
        near = G.run(alpha=0.15, R=40, seed=9, topk=8, src_begin=n - 3000, src_end=n, stats=True, **kw)
        for a, b in zip((*far.sparse_rows(), *far.topk()), (*near.sparse_rows(), *near.topk())):
            assert np.array_equal(a, b)
        assert far.info().steps == near.info().steps
        far.free()
        near.free()
    G.free()
