"""Work chunks of the persistent walker at the limits of what a warp takes at
once (31 whole sources, parts of 32), against one thread per walk."""
import numpy as np
import pytest

from paper_1903_11749_gb300 import inputs as I
from test_gpu_parity import ctx, ppr  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("R", [1, 3, 12, 13, 100])
@pytest.mark.parametrize("wide", [False, True])
def test_every_chunk_size_walks_the_same(ppr, ctx, R, wide):  # noqa: F811
    g = I.random_small_graph(3000, 14000, seed=8, wmax=(1 << 31) if wide else 50, dangling=100)
    G = ctx.load_graph(g.n, g.row_ptr, g.col, g.w)
    src = np.random.default_rng(5).integers(0, g.n, 2971).astype(np.int32)
    for S in (33, 2971):
        ref = G.run_list(src[:S], alpha=0.15, R=R, seed=4, topk=5, kernel=1)
        want = (*ref.sparse_rows(), *ref.topk())
        for cs in (0, 1, 31, 32, 500):
            r = G.run_list(src[:S], alpha=0.15, R=R, seed=4, topk=5, chunk_sources=cs)
            for a, b in zip((*r.sparse_rows(), *r.topk()), want):
                assert np.array_equal(a, b)
            r.free()
        ref.free()
    G.free()
