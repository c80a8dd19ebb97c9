"""The serving loop's ring of 64 slots reused many times within a burst, by
queries of every size of R that the loop's reductions tell apart (one to
1,024: registers up to 128, shared memory above; walking warps help up to
128).  Each answer must equal the rows of an ordinary run over its sources."""
import threading

import numpy as np
import pytest

from paper_1903_11749_gb300 import inputs as I
from paper_1903_11749_gb300 import ppr

pytestmark = pytest.mark.gpu

RS = [1, 2, 31, 33, 64, 100, 128, 129, 200, 256, 257, 1000, 1024]


@pytest.fixture(scope="module")
def graphs():
    """The same edges with 32-bit and with 64-bit row totals."""
    ctx = ppr.Context(0)
    loaded = [I.random_small_graph(6000, 60000, seed=51, wmax=wmax, dangling=60) for wmax in (50, 1 << 31)]
    return ctx, [ctx.load_graph(g.n, g.row_ptr, g.col, g.w) for g in loaded]


@pytest.fixture(scope="module")
def graph(graphs):
    return graphs[0], graphs[1][0]


@pytest.mark.parametrize("smax,count", [(8, 600), (700, 200)])
@pytest.mark.parametrize("wide,sampler", [(0, 0), (0, 1), (1, 0)])
def test_slots_reused_within_a_burst(graphs, smax, count, wide, sampler):
    ctx, G = graphs[0], graphs[1][wide]
    assert G.info().wide == wide
    want = {R: G.run(alpha=0.15, R=R, seed=R, topk=8, sampler=sampler).topk() for R in RS}
    rng = np.random.default_rng(7)
    qs = [(RS[i % len(RS)], rng.integers(0, 6000, int(rng.integers(1, smax + 1))).astype(np.int32))
          for i in range(count)]
    ctx.serve_start(G, max_sources=smax, max_topk=8, memory_budget=64 << 20, sampler=sampler)
    try:
        ids = [None] * count

        def submitter(first):
            for i in range(first, count, 2):
                ids[i] = ctx.submit(qs[i][1], alpha=0.15, R=qs[i][0], seed=qs[i][0], topk=8)

        threads = [threading.Thread(target=submitter, args=(k,)) for k in range(2)]
        for t in threads:
            t.start()
        for t in threads:
            t.join()
        for i, (R, src) in enumerate(qs):
            idx, cnt, _ = ctx.poll(ids[i], len(src), 8, timeout_ms=60000)
            assert np.array_equal(idx, want[R][0][src]) and np.array_equal(cnt, want[R][1][src]), (i, R)
        info = ctx.serve_info()
        assert info["completed"] == count and info["in_flight"] == 0
        assert info["reduced"] == sum(len(s) for _, s in qs)
    finally:
        ctx.serve_stop()


def test_queries_published_while_the_walkers_leave(graph):
    """With an idle time of a microsecond the loop ends at once whenever nothing
    is in flight.  Queries that arrive while an earlier one is still being
    reduced (R above what walking warps help with, so they have nothing to do)
    or just as the warps leave are walked all the same, here or by the next
    launch; none waits for the bound on queries in flight."""
    import time
    ctx, G = graph
    want = {R: G.run(alpha=0.15, R=R, seed=R, topk=8).topk() for R in (40, 1000)}
    rng = np.random.default_rng(3)
    ctx.serve_start(G, max_sources=6000, max_topk=8, memory_budget=256 << 20, idle_us=1)
    try:
        for delay in np.linspace(0, 6e-3, 40):
            work = []
            for R, ns, pause in ((1000, 6000, delay), (40, 50, delay / 7), (40, 3, 0)):
                src = rng.integers(0, 6000, ns).astype(np.int32)
                work.append((R, src, ctx.submit(src, alpha=0.15, R=R, seed=R, topk=8)))
                time.sleep(pause)
            for R, src, q in work:
                idx, cnt, _ = ctx.poll(q, len(src), 8, timeout_ms=20000)
                assert np.array_equal(idx, want[R][0][src]) and np.array_equal(cnt, want[R][1][src])
        for i in range(400):  # one small query at a time, at any moment of the loop's end
            src = rng.integers(0, 6000, 3).astype(np.int32)
            q = ctx.submit(src, alpha=0.15, R=40, seed=40, topk=8)
            idx, cnt, _ = ctx.poll(q, 3, 8, timeout_ms=20000)
            assert np.array_equal(idx, want[40][0][src]) and np.array_equal(cnt, want[40][1][src])
            time.sleep((i % 50) * 2e-6)
        info = ctx.serve_info()
        assert info["launches"] > 1 and info["in_flight"] == 0
    finally:
        ctx.serve_stop()


def test_warps_without_work_sleep(graph):
    """While a few warps walk one query for a long time, those without work
    sleep most of the time (up to 33 us between looks that take a few), so
    that they do not stand in the way of the query's reads and counts."""
    import time
    ctx, G = graph

    def ended():
        deadline = time.time() + 20
        while ctx.serve_info()["running"] and time.time() < deadline:
            time.sleep(0.005)
        return ctx.serve_info()

    ctx.serve_start(G, max_sources=8, max_topk=8, memory_budget=64 << 20, idle_us=10_000)
    try:
        before = ended()
        # 1,024 walks (32 warps' worth) of 20,000 steps on average
        q = ctx.submit(np.array([5], np.int32), alpha=5e-5, R=1024, seed=1, topk=8)
        ctx.poll(q, 1, 8, timeout_ms=60000)
        after = ended()
        slept = after["cycles_sleep"] - before["cycles_sleep"]
        assert slept > 0.5 * (after["cycles_total"] - before["cycles_total"])
    finally:
        ctx.serve_stop()


def test_a_small_query_does_not_wait_for_the_reductions_of_large_ones(graph):
    """Eight queries of 6,000 sources with R 1,000 leave tens of milliseconds of
    reductions; a query of three sources published when the first of them is
    done is answered in well under half of what is left of that."""
    ctx, G = graph
    want = G.run(alpha=0.15, R=1000, seed=1, topk=8).topk()
    large, small = np.arange(6000, dtype=np.int32), np.array([5, 17, 4000], np.int32)
    ctx.serve_start(G, max_sources=6000, max_topk=8, memory_budget=512 << 20)
    try:
        for _ in range(2):  # (the first time warms up)
            ids = [ctx.submit(large, alpha=0.15, R=1000, seed=1, topk=8) for _ in range(8)]
            got = [ctx.poll(ids[0], 6000, 8, timeout_ms=60000)]
            q = ctx.submit(small, alpha=0.15, R=1000, seed=1, topk=8)
            idx, cnt, st = ctx.poll(q, 3, 8, timeout_ms=60000)
            got += [ctx.poll(i, 6000, 8, timeout_ms=60000) for i in ids[1:]]
        assert np.array_equal(idx, want[0][small]) and np.array_equal(cnt, want[1][small])
        for a, b, _ in got:
            assert np.array_equal(a, want[0]) and np.array_equal(b, want[1])
        last = max(s["done_ns"] for _, _, s in got)
        assert last > st["submit_ns"]
        assert st["done_ns"] - st["submit_ns"] < 0.5 * (last - st["submit_ns"])
    finally:
        ctx.serve_stop()
