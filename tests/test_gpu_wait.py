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


def test_a_finished_run_is_waited_for_beside_large_output_copies():
    """Runs that are over are waited for while another thread's ppr_run_to_host
    copies rows: the wait neither queues behind those copies (each takes more
    than ten milliseconds here) nor overruns its timeout of 0."""
    import time

    import torch

    n, R = 1 << 18, 1500
    g = I.er_graph(n, 1 << 22, 1, 10, seed=5)
    small = I.er_graph(2000, 16000, 1, 10, seed=5)
    ctx = ppr.Context(0)
    H = ctx.load_graph(g.n, g.row_ptr, g.col, g.w)
    G = ctx.load_graph(small.n, small.row_ptr, small.col, small.w)
    rows = [torch.zeros(n + 1, dtype=torch.int64, pin_memory=True)] + [
        torch.zeros(n * R, dtype=torch.int32, pin_memory=True) for _ in range(2)]
    H.run_to_host(*rows, alpha=0.15, R=R, seed=3, parts=1)
    runs = [G.run(alpha=0.15, R=10, topk=4, src_end=50, wait=False) for _ in range(60)]
    torch.cuda.synchronize()
    busy = []

    def host():
        t = time.perf_counter()
        for _ in range(3):
            H.run_to_host(*rows, alpha=0.15, R=R, seed=3, parts=1)
        busy.append(time.perf_counter() - t)

    th = threading.Thread(target=host)
    th.start()
    waits = []
    for r in runs:
        if not th.is_alive():
            break
        t = time.perf_counter()
        r.wait(0)
        waits.append(time.perf_counter() - t)
        time.sleep(0.001)
    th.join()
    assert busy[0] > 0.03 and len(waits) > 10
    assert sorted(waits)[-2] < 0.003, sorted(waits)[-5:]  # (one may have been descheduled)
    want = runs[0].info().steps
    assert want > 0 and all(r.info().steps == want for r in runs[: len(waits)])


def test_more_unread_runs_than_words():
    """More runs than there are words for their counters (1,024), some of them
    freed before they end: every step count is the run's own."""
    g = I.er_graph(2000, 16000, 1, 10, seed=5)
    ctx = ppr.Context(0)
    G = ctx.load_graph(g.n, g.row_ptr, g.col, g.w)

    def start(i):
        return G.run(alpha=0.15, R=8 + i % 5, seed=i % 7, src_end=100, wait=False)

    want = [start(i).wait().info().steps for i in range(35)]
    for _ in range(2):
        runs = [start(i) for i in range(1400)]
        for r in runs[::3]:
            r.free()
        runs += [start(i) for i in range(1400, 1900)]
        for i, r in enumerate(runs):
            if r.h:
                assert r.wait().info().steps == want[i % 35]
                r.free()
    start(0).free()  # (the context goes with a run in flight)


def test_a_context_closes_beside_a_busy_serving_loop():
    """Another context's resident loop keeps the device busy with one long query;
    contexts that have read runs are closed meanwhile without waiting for it."""
    import time

    g = I.random_small_graph(6000, 60000, seed=51, wmax=50, dangling=60)
    one = ppr.Context(0)
    G = one.load_graph(g.n, g.row_ptr, g.col, g.w)
    used = []
    for _ in range(3):
        c = ppr.Context(0)
        H = c.load_graph(g.n, g.row_ptr, g.col, g.w)
        H.run(alpha=0.2, R=8, src_end=10).free()
        H.free()
        used.append(c)
    one.serve_start(G)
    try:
        q = one.submit(np.array([3], np.int32), alpha=2e-5, R=1000, seed=1, topk=4)  # walks of 50,000 steps
        time.sleep(0.01)
        t0 = time.perf_counter()
        for c in used:
            c.close()
        closed = time.perf_counter() - t0
        one.poll(q, 1, 4, timeout_ms=60000)
        answered = time.perf_counter() - t0
        assert answered > 0.05 and closed < 0.2 * answered
    finally:
        one.serve_stop()
