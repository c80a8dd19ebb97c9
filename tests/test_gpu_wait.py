"""Waiting for runs and reading them from several threads of one context, and
the limits of the wait's timeout."""
import ctypes as C
import threading

import numpy as np
import pytest

from paper_1903_11749_gb300 import inputs as I
from paper_1903_11749_gb300 import ppr

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def graph():
    g = I.er_graph(2000, 16000, 1, 10, seed=5)
    ctx = ppr.Context(0)
    return ctx.load_graph(g.n, g.row_ptr, g.col, g.w)


@pytest.mark.parametrize("timeout_ms", [1 << 40, 1 << 62, (1 << 63) - 1])
def test_wait_takes_any_timeout(graph, timeout_ms):
    """A long timeout is a long timeout, whatever unit the wait counts in."""
    r = graph.run(alpha=0.15, R=4000, seed=1, topk=8, wait=False)
    assert ppr.lib().ppr_wait(r.h, C.c_int64(timeout_ms)) == 0
    r.free()


@pytest.mark.parametrize("threads", [2, 8])
def test_results_of_several_threads(graph, threads):
    """Threads that wait for and read runs of their own at the same time get
    their own step counts and rows."""
    def query(seed):
        r = graph.run(alpha=0.15, R=16 + seed, seed=seed, topk=8, src_begin=0, src_end=100 + 50 * seed)
        rows = r.sparse_rows()
        steps = r.info().steps
        r.free()
        return [np.int64(steps), *rows]

    want = [query(t) for t in range(threads)]
    got = [[] for _ in range(threads)]

    def work(t):
        for _ in range(60):
            got[t].append(query(t))

    ts = [threading.Thread(target=work, args=(t,)) for t in range(threads)]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    for t in range(threads):
        assert len(got[t]) == 60
        for g in got[t]:
            assert all(np.array_equal(a, b) for a, b in zip(g, want[t]))
