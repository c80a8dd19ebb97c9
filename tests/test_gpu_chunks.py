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


@pytest.mark.parametrize("R", [1, 8, 13, 50, 4096])
def test_autotune_returns_a_chunk_that_is_used(ppr, ctx, R):  # noqa: F811
    """No chunk beyond the 31 sources a warp takes at once is timed or
    returned, and each is timed once (two block sizes, then four refills)."""
    g = I.random_small_graph(3000, 14000, seed=8, wmax=50, dangling=100)
    G = ctx.load_graph(g.n, g.row_ptr, g.col, g.w)
    t = G.autotune(alpha=0.15, R=R, sample_sources=400)
    base = min(31, max(1, 400 // R))
    chunks = {min(31, c, (1 << 19) // R) for c in (max(1, base // 4), max(1, base // 2), base, 2 * base, 4 * base)}
    assert t["chunk_sources"] in chunks
    assert t["candidates"] == 2 * len(chunks) + 4
    G.free()


@pytest.mark.parametrize("kernel", [0, 1])
def test_autotune_times_small_chunks_of_a_batch(ppr, ctx, kernel):  # noqa: F811
    """A batch's chunk table grows as chunks shrink: the tuner's scratch holds
    the largest, whatever kernel the run asks for."""
    inst = I.chung_lu_instances(count=20, nmin=50, nmax=800, seed=6)
    G = ctx.load_graph_batch(inst.node_off, inst.row_ptr, inst.col, inst.w)
    t = G.autotune(sample_sources=2000, alpha=0.15, R=20, seed=1, kernel=kernel)
    assert t["candidates"] == 2 * len({5, 10, 20, 31}) + 4 and t["ms"] > 0 and t["chunk_sources"] in (5, 10, 20, 31)
    G.free()
