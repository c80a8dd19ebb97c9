"""The walk layout's guide slots against the oracle where they can go wrong:
degrees on both sides of every class limit, rows whose first edge starts
anywhere within a 32-byte sector, ranges with exactly as many edges as a slot
holds and one more, runs of light edges beside heavy ones (overflow over one
sector, five, and hundreds), row totals just below and above 2^32, and wide
rows whose ranges are 32 bits long.  Counts are integers: every comparison is
exact."""
import numpy as np
import pytest

from paper_1903_11749_gb300 import inputs as I
from test_gpu_parity import assert_same, oracle_rows

pytestmark = pytest.mark.gpu

DEGREES = [0, 1, 2, 3, 4, 5, 7, 8, 9, 15, 16, 17, 31, 32, 33, 63, 65, 127, 129, 1000, 4095, 4097, 9000]


@pytest.fixture(scope="module")
def ppr():
    from paper_1903_11749_gb300 import build as B
    B.build()
    from paper_1903_11749_gb300 import ppr as P
    return P


@pytest.fixture(scope="module")
def ctx(ppr):
    return ppr.Context(0)


def weights(style, d, rng):
    if style == "equal":
        return np.full(d, 3)
    if style == "light_runs":  # a few heavy edges among many light ones: hundreds of edges in a range
        w = np.full(d, 2)
        if d > 8:
            w[rng.choice(d, size=max(1, d // 100), replace=False)] = 4000
        return w
    if style == "near_2_32":  # narrow, totals close to 2^32
        return np.full(d, max(1, (2**32 - 1) // max(d, 1)))
    if style == "one_giant":  # wide from one edge; the others share the rest
        w = rng.integers(1, 2**20, size=d)
        if d:
            w[d // 2] = 2**32 - 1
        return w
    assert style == "all_giant"  # ranges of 2^32 - 1
    return np.full(d, 2**32 - 1)


def graph(style, seed):
    rng = np.random.Generator(np.random.PCG64(seed))
    deg = np.array([d for d in DEGREES for _ in range(4)])
    rng.shuffle(deg)
    n = len(deg)
    rp = np.zeros(n + 1, dtype=np.int64)
    np.cumsum(deg, out=rp[1:])
    # half of the targets among the long rows, so that walks meet them
    long_rows = np.flatnonzero(deg >= 63)
    col = np.where(rng.random(rp[-1]) < 0.5, rng.choice(long_rows, size=rp[-1]), rng.integers(0, n, size=rp[-1]))
    w = np.concatenate([weights(style, int(d), rng) for d in deg])
    return I.Graph(n, rp, col.astype(np.int32), w.astype(np.uint32))


@pytest.mark.parametrize("style", ["equal", "light_runs", "near_2_32", "one_giant", "all_giant"])
def test_rows_at_every_class_limit(ppr, ctx, oracle, style):
    g = graph(style, seed=11)
    for renumber in (False, True):
        G = ctx.load_graph(g.n, g.row_ptr, g.col, g.w, renumber=renumber)
        assert G.info().wide == (1 if style.endswith("giant") else 0)
        for kw in (dict(dangling=0), dict(dangling=1), dict(segments=True)):
            ref = oracle_rows(oracle, g, 0.15, 500, 3, topk=8, **kw)
            for kernel in (ppr.KERNEL_PERSISTENT, ppr.KERNEL_PLAIN):
                assert_same(G.run(alpha=0.15, R=500, seed=3, topk=8, kernel=kernel, **kw), ref, topk=8)
            if style == "light_runs":  # the statistics launch walks the same draws
                r = G.run(alpha=0.15, R=500, seed=3, topk=8, stats=True, **kw)
                assert_same(r, ref, topk=8)
                assert 0 < r.info().sectors
        G.free()


def test_instances_with_and_without_edges(ppr, ctx, oracle):
    """Rows of different instances share sectors and tiles; an instance may have no edge at all."""
    parts = [graph("light_runs", 5), I.from_edges(3, []), graph("equal", 6), I.from_edges(1, [(0, 0, 7)]),
             I.random_small_graph(40, 90, seed=4, dangling=3)]
    off = np.concatenate([[0], np.cumsum([p.n for p in parts])]).astype(np.int64)
    rp = np.concatenate([[0], np.cumsum(np.concatenate([np.diff(p.row_ptr) for p in parts]))]).astype(np.int64)
    col = np.concatenate([p.col for p in parts]).astype(np.int32)
    w = np.concatenate([p.w for p in parts]).astype(np.uint32)
    G = ctx.load_graph_batch(off, rp, col, w)
    res = G.run(alpha=0.2, R=100, seed=2, topk=5)
    rows, rc, rn = res.sparse_rows()
    idx, cnt = res.topk(5)
    for t, p in enumerate(parts):
        ref = oracle_rows(oracle, p, 0.2, 100, 2, tag=t, topk=5)
        a, b = rows[off[t]], rows[off[t + 1]]
        orp, oc, on = ref["rows"]
        assert np.array_equal(rows[off[t]: off[t + 1] + 1] - a, orp)
        assert np.array_equal(rc[a:b], oc) and np.array_equal(rn[a:b], on)
        assert np.array_equal(idx[off[t]: off[t + 1]], ref["topk"][0])
        assert np.array_equal(cnt[off[t]: off[t + 1]], ref["topk"][1])
    G.free()


@pytest.mark.parametrize("bad", ["weight", "col"])
def test_invalid_edges_are_still_refused(ppr, ctx, bad):
    g = graph("equal", 8)
    col, w = g.col.copy(), g.w.copy()
    if bad == "weight":
        w[len(w) // 2] = 0
    else:
        col[len(col) // 3] = g.n
    with pytest.raises(ppr.PPRError) as e:
        ctx.load_graph(g.n, g.row_ptr, col, w)
    assert e.value.code == ppr.PPR_EINVAL


@pytest.mark.parametrize("kernel", [0, 1])
@pytest.mark.parametrize("segments", [False, True])
def test_flat_model_counts_the_node_a_walk_ends_at(ppr, ctx, kernel, segments):
    """In dangling mode 1 a walk that comes to a node without out-edges ends
    there; the flat-CSR model reads one sector to find that out.  Here every
    walk makes one draw at a row of 16 edges (row_ptr, three probe sectors, the
    target) and ends at node 100; walks from node 100 make none."""
    n, d, R = 101, 16, 50
    rp = np.minimum(np.arange(n + 1, dtype=np.int64), n - 1) * d
    G = ctx.load_graph(n, rp, np.full(d * (n - 1), n - 1, np.int32), np.ones(d * (n - 1), np.uint32))
    r = G.run(alpha=1e-7, R=R, seed=1, dangling=1, stats=True, kernel=kernel, segments=segments)
    i = r.info()
    assert i.steps == (n - 1) * R
    assert i.model_sectors == (n - 1) * R * (1 + 3 + 1) + n * R
