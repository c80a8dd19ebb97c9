"""The measured work of the Monte Carlo PPR library: calls a user's program
makes through the Python binding (paper_1903_11749_gb300.ppr), over the range
of graphs, walk counts, samplers and layouts it is used with.

Graphs are made on the GPU from the seed alone, with the shapes of the
repository's own workloads: R-MAT (a .57, b .19, c .19, 16 edges a node, about
5 % dangling nodes, Zipf(1.5) weights on [1, 1000]), Chung-Lu (exponent 2.3,
mean degree 12, weights U[1, 100]) and uniform random graphs (weights
U[1, 10]).  Every output is a whole number (node ids and counts), so nothing
here has a value in floating point to be compared with.
"""
import math

import torch

from paper_1903_11749_gb300 import ppr

DEV = "cuda"
_ctx = None


def _context():
    global _ctx
    if _ctx is None:
        _ctx = ppr.Context(0)
    return _ctx


# ------------------------------------------------------------------- cases ----

def listed():
    return [
        # a small multi-source query on a resident graph: answered in
        # microseconds, so launches and latency are what it costs
        {"name": "query_small", "kind": "list", "graph": "rmat", "scale": 18, "sources": 64, "R": 100, "topk": 32,
         "alpha": 0.15, "sampler": 0, "dangling": 0},
        # the whole job on a tiny graph: load the CSR, 1,000 walks a node, rows
        {"name": "er1k_job", "kind": "job", "graph": "er", "n": 1000, "m": 10000, "R": 1000, "topk": 32,
         "alpha": 0.15, "sampler": 0, "segments": False, "dangling": 0},
        # few sources with as many walks as the library takes and a long top-k:
        # rankings that are to be accurate (the accuracy workload)
        {"name": "accurate_rankings", "kind": "list", "graph": "chunglu", "n": 50000, "sources": 500, "R": 4096,
         "topk": 1000, "alpha": 0.15, "sampler": 0, "dangling": 0},
        # the whole job at scale 20: load, 100 walks a node, rows and top-32
        {"name": "rmat20_job", "kind": "job", "graph": "rmat", "scale": 20, "R": 100, "topk": 32, "alpha": 0.2,
         "sampler": 0, "segments": False, "dangling": 0},
        # every source of a resident scale-20 graph with alias tables, into the
        # caller's own buffers
        {"name": "rmat20_alias", "kind": "into", "graph": "rmat", "scale": 20, "R": 100, "topk": 32, "alpha": 0.2,
         "sampler": 1, "segments": False, "dangling": 0},
        # CSR from page-locked host memory, rows and top-k back into it
        {"name": "rmat19_host", "kind": "host", "graph": "rmat", "scale": 19, "R": 100, "topk": 32, "alpha": 0.2,
         "sampler": 0, "segments": False, "dangling": 0},
        # weights as amounts (row totals above 32 bits: the wide layout), walks
        # that end at nodes without out-edges
        {"name": "amounts_wide", "kind": "into", "graph": "rmat", "scale": 18, "R": 100, "topk": 32, "alpha": 0.15,
         "sampler": 0, "segments": False, "dangling": 1, "wmax": 10000000},
        # many uneven graphs in one launch
        {"name": "batch_graphs", "kind": "batch", "graph": "chunglu_batch", "count": 256, "nmin": 100, "nmax": 50000,
         "R": 200, "topk": 32, "alpha": 0.15, "sampler": 0, "dangling": 0},
        # a burst of queries of very different sizes through the serving loop
        {"name": "serve_burst", "kind": "serve", "graph": "rmat", "scale": 20, "queries": 64, "smax": 20000, "R": 100,
         "topk": 32, "alpha": 0.15, "sampler": 0},
        # the whole job at scale 24, far beyond L2, with a hub of over 10^6 edges
        {"name": "rmat24_job", "kind": "job", "graph": "rmat", "scale": 24, "R": 50, "topk": 64, "alpha": 0.15,
         "sampler": 0, "segments": False, "dangling": 0, "hub": 1200000},
        # a quarter of its sources with the depth-3 segment tables (a job split
        # over source ranges keeps the graph and its tables)
        {"name": "rmat24_segments", "kind": "range", "graph": "rmat", "scale": 24, "part": 4, "R": 50, "topk": 64,
         "alpha": 0.15, "sampler": 0, "segments": True, "dangling": 0, "hub": 1200000},
        # the same with alias tables
        {"name": "rmat24_alias", "kind": "range", "graph": "rmat", "scale": 24, "part": 4, "R": 50, "topk": 64,
         "alpha": 0.15, "sampler": 1, "segments": False, "dangling": 0, "hub": 1200000},
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["list", "list", "job", "job", "into", "into", "range", "host", "batch", "serve"])
    alpha = rng.choice([0.1, 0.15, 0.2, 0.5])
    topk = rng.choice([1, 10, 32, 64, 100])
    sampler = rng.choice([0, 0, 1])
    c = {"kind": kind, "alpha": alpha, "topk": topk, "sampler": sampler}
    if kind == "serve":
        return {**c, "graph": "rmat", "scale": rng.randint(16, 21), "queries": rng.randint(8, 64),
                "smax": _log_int(rng, 100, 30000), "R": _log_int(rng, 20, 200)}
    c["dangling"] = rng.choice([0, 0, 0, 1])
    if kind == "batch":
        return {**c, "graph": "chunglu_batch", "count": _log_int(rng, 3, 300), "nmin": rng.choice([20, 100, 700]),
                "nmax": rng.choice([3000, 20001, 50000]), "R": _log_int(rng, 20, 400)}
    if kind == "list":
        c["sources"] = _log_int(rng, 1, 5000)
        c["R"] = _log_int(rng, 16, 4096)
        c["topk"] = rng.choice([1, 10, 32, 100, 1000])
        if rng.random() < 0.5:
            return {**c, "graph": "chunglu", "n": _log_int(rng, 500, 200000)}
        return {**c, "graph": "rmat", "scale": rng.randint(14, 22)}
    c["segments"] = sampler == 0 and rng.random() < 0.25
    if kind == "range":
        return {**c, "graph": "rmat", "scale": 24, "part": rng.randint(3, 40), "R": _log_int(rng, 10, 60),
                "hub": rng.choice([0, 300000, 1200000])}
    if kind == "host":
        return {**c, "graph": "rmat", "scale": rng.randint(14, 19), "R": _log_int(rng, 10, 130)}
    if rng.random() < 0.3:
        n = _log_int(rng, 100, 30000)
        return {**c, "graph": "er", "n": n, "m": n * rng.randint(2, 40), "R": _log_int(rng, 20, 1000)}
    if rng.random() < 0.4:
        return {**c, "graph": "chunglu", "n": _log_int(rng, 1000, 400000), "R": _log_int(rng, 16, 300)}
    c = {**c, "graph": "rmat", "scale": rng.randint(12, 21), "R": _log_int(rng, 10, 130)}
    if sampler == 0 and rng.random() < 0.5:  # (alias tables are for row totals below 2^32)
        c["wmax"] = 10000000
    return c


# ------------------------------------------------------------------ graphs ----

def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    return g


def _csr(n, src, dst, w):
    """CSR (row_ptr int64[n + 1], col int32[m], w uint32 as int32[m]) of edge triples, on the GPU."""
    src, order = torch.sort(src, stable=True)
    col = dst[order]
    row_ptr = torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    row_ptr[1:] = torch.searchsorted(src, torch.arange(n, dtype=src.dtype, device=DEV), right=True)
    return row_ptr, col.to(torch.int32).contiguous(), w[order].to(torch.int32).contiguous()


def _zipf(count, g, wmax, s=1.5):
    """Weights with P(k) ~ k^-s on {1 .. wmax}; amounts (a large wmax) are log-uniform instead."""
    if wmax > 100000:
        u = torch.rand(count, generator=g, device=DEV, dtype=torch.float64)
        return torch.exp(u * math.log(wmax)).to(torch.int32).clamp_(1, wmax)
    cdf = torch.cumsum(torch.arange(1, wmax + 1, dtype=torch.float64, device=DEV) ** -s, 0)
    cdf = (cdf / cdf[-1]).to(torch.float32)
    u = torch.rand(count, generator=g, device=DEV)
    return torch.searchsorted(cdf, u, right=True).clamp_(max=wmax - 1).to(torch.int32) + 1


def _rmat(scale, seed, hub=0, wmax=1000):
    n, m, g = 1 << scale, 16 << scale, _gen(seed)
    src = torch.zeros(m, dtype=torch.int32, device=DEV)
    dst = torch.zeros(m, dtype=torch.int32, device=DEV)
    for _ in range(scale):
        bit = torch.rand(m, generator=g, device=DEV) < 0.24  # c + d
        r = torch.rand(m, generator=g, device=DEV)
        dbit = torch.where(bit, r < 0.05 / 0.24, r < 0.19 / 0.76)
        src = src * 2 + bit
        dst = dst * 2 + dbit
        del bit, r, dbit
    if hub:
        src[torch.rand(m, generator=g, device=DEV) < hub / m] = 0
    deg = torch.bincount(src, minlength=n)
    empty = torch.nonzero(deg == 0).flatten()
    keep = torch.rand(empty.numel(), generator=g, device=DEV) < 0.05 * n / max(1, empty.numel())
    extra = empty[~keep].to(torch.int32)
    src = torch.cat([src, extra])
    dst = torch.cat([dst, torch.randint(0, n, (extra.numel(),), generator=g, device=DEV, dtype=torch.int32)])
    return (n,) + _csr(n, src, dst, _zipf(src.numel(), g, wmax))


def _power_nodes(count, n, g, exponent=2.3):
    """Nodes of [0, n) drawn in proportion to (i + 1)^(-1 / (exponent - 1)); n a number or a tensor."""
    q = 1.0 - 1.0 / (exponent - 1.0)
    u = torch.rand(count, generator=g, device=DEV, dtype=torch.float64)
    i = ((u * ((n + 1.0) ** q - 1.0) + 1.0) ** (1.0 / q) - 1.0).to(torch.int64)
    return torch.minimum(i, torch.as_tensor(n, device=DEV).to(torch.int64) - 1).clamp_(min=0)


def _chunglu(n, seed):
    g, m = _gen(seed), 12 * n
    src, dst = _power_nodes(m, float(n), g), _power_nodes(m, float(n), g)
    return (n,) + _csr(n, src, dst, torch.randint(1, 101, (m,), generator=g, device=DEV))


def _chunglu_batch(count, nmin, nmax, seed):
    """count graphs side by side: node offsets, and a CSR whose targets count within their graph."""
    g = _gen(seed)
    # sizes log-uniform on [nmin, nmax] in a mixed order, the same for every seed (so that outputs keep their shapes)
    u = ((torch.arange(count, dtype=torch.float64) * 0.6180339887498949) % 1.0).to(DEV)
    ns = torch.exp(math.log(nmin) + u * math.log(nmax / nmin)).to(torch.int64)
    off = torch.zeros(count + 1, dtype=torch.int64, device=DEV)
    off[1:] = torch.cumsum(ns, 0)
    which = torch.repeat_interleave(torch.arange(count, device=DEV), 12 * ns)
    size = ns[which].to(torch.float64)
    src = _power_nodes(which.numel(), size, g) + off[which]
    dst = _power_nodes(which.numel(), size, g)
    n = int(off[-1])
    return (off.cpu().numpy(), n) + _csr(n, src, dst, torch.randint(1, 101, (which.numel(),), generator=g, device=DEV))


def _graph(case, seed):
    if case["graph"] == "rmat":
        return _rmat(case["scale"], seed, case.get("hub", 0), case.get("wmax", 1000))
    if case["graph"] == "chunglu":
        return _chunglu(case["n"], seed)
    g, n, m = _gen(seed), case["n"], case["m"]
    ends = torch.randint(0, n, (2, m), generator=g, device=DEV)
    return (n,) + _csr(n, ends[0], ends[1], torch.randint(1, 11, (m,), generator=g, device=DEV))


# --------------------------------------------------------------- the calls ----

class _State:
    pass


class _Server(_State):
    """A context of its own that serves; the loop gives the GPU back after a millisecond without work."""

    def __init__(self, graph, case):
        n, rp, col, w = graph
        self.ctx = ppr.Context(0)
        self.G = self.ctx.load_graph(n, rp, col, w)
        self.ctx.serve_start(self.G, max_sources=case["smax"], max_topk=case["topk"], sampler=case["sampler"],
                             memory_budget=2 << 30, idle_us=1000)

    def __del__(self):
        self.ctx.serve_stop()
        self.G.free()
        self.ctx.close()


def _out(S, topk):
    return (torch.zeros((S, topk), dtype=torch.int32, device=DEV), torch.zeros((S, topk), dtype=torch.int32, device=DEV))


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        off, n, rp, col, w = _chunglu_batch(case["count"], case["nmin"], case["nmax"], seed)
    else:
        n, rp, col, w = _graph(case, seed)
    R, topk = case["R"], case["topk"]
    if kind == "serve":
        s = _Server((n, rp, col, w), case)
        g = _gen(seed + 1)
        # sizes log-uniform on [1, smax] in a mixed order, the same for every seed
        sizes = [max(1, int(math.exp((i * 0.6180339887498949) % 1.0 * math.log(case["smax"])))) for i in range(case["queries"])]
        s.queries = [torch.randint(0, n, (k,), generator=g, device=DEV, dtype=torch.int32).cpu().numpy() for k in sizes]
        s.case, s.seed = case, seed
        return s
    s = _State()
    s.case, s.n = case, n
    s.run = dict(alpha=case["alpha"], R=R, seed=seed, topk=topk, sampler=case["sampler"], dangling=case["dangling"],
                 segments=case.get("segments", False))
    ctx = s.ctx = _context()
    if kind == "host":
        s.csr = [t.cpu().pin_memory() for t in (rp, col, w)]
        cap = min(R, n) * n
        s.rows = [torch.zeros(n + 1, dtype=torch.int64, pin_memory=True)] + [
            torch.zeros(cap, dtype=torch.int32, pin_memory=True) for _ in range(2)]
        s.top = [torch.zeros((n, topk), dtype=torch.int32, pin_memory=True) for _ in range(2)]
        return s
    if kind == "job":
        s.csr = [rp, col, w]
        s.m = int(col.numel())
    else:
        s.G = ctx.load_graph_batch(off, rp, col, w) if kind == "batch" else ctx.load_graph(n, rp, col, w, m=int(col.numel()))
    S = n
    if kind == "range":
        S = n // case["part"]
        s.run.update(src_begin=(case["part"] // 2) * S, src_end=(case["part"] // 2) * S + S)
    if kind == "list":
        S = case["sources"]
        s.sources = torch.randint(0, n, (S,), generator=_gen(seed + 1), device=DEV, dtype=torch.int32).cpu().numpy()
    s.S, s.top = S, _out(S, topk)
    cap = min(R, n)
    if kind in ("job", "range"):
        s.rows = [torch.zeros(S + 1, dtype=torch.int64, device=DEV)] + [
            torch.zeros(S * cap, dtype=torch.int32, device=DEV) for _ in range(2)]
    if kind in ("into", "batch"):
        if kind == "into" and (s.run["sampler"] == 1 or s.run["segments"]):
            # the tables of the sampler are built by an ordinary run
            s.G.run(**{**s.run, "src_begin": 0, "src_end": 1}).free()
        if kind == "batch":
            if s.run["sampler"] == 1:
                s.G.run(**{**s.run, "src_begin": 0, "src_end": 1}).free()
            cap = min(R, int((off[1:] - off[:-1]).max()))
        s.cap = cap
        s.work = torch.empty(s.G.workspace_size(**s.run), dtype=torch.uint8, device=DEV)
        s.nnz = torch.zeros(S, dtype=torch.int32, device=DEV)
        s.rows = [torch.zeros((S, cap), dtype=torch.int32, device=DEV) for _ in range(2)]
    return s


def run(s):
    c = s.case
    kind = c["kind"]
    if kind == "serve":
        ids = [s.ctx.submit(q, alpha=c["alpha"], R=c["R"], seed=s.seed + i, topk=c["topk"])
               for i, q in enumerate(s.queries)]
        got = [s.ctx.poll(i, len(q), c["topk"])[:2] for i, q in zip(ids, s.queries)]
        # one answer a query, all in one pair of arrays
        return [torch.cat([torch.from_numpy(x[k].astype("int32", copy=False)) for x in got]) for k in (0, 1)]
    if kind == "host":
        rp, col, w = s.csr
        G = s.ctx.load_graph(s.n, rp, col, w, m=int(col.numel()))
        nnz, _ = G.run_to_host(s.rows[0], s.rows[1], s.rows[2], s.top[0], s.top[1], **s.run)
        G.free()
        return [nnz, *s.rows, *s.top]
    if kind in ("into", "batch"):
        s.G.run_into(s.work, s.nnz, s.rows[0], s.rows[1], s.cap, s.top[0], s.top[1], **s.run)
        return [s.nnz, *s.rows, *s.top]
    if kind == "list":
        r = s.G.run_list(s.sources, **s.run)
        r.topk_into(c["topk"], *s.top)
        steps = r.info().steps
        r.free()
        return [steps, *s.top]
    G = s.ctx.load_graph(s.n, *s.csr, m=s.m) if kind == "job" else s.G
    r = G.run(**s.run)
    nnz = r.sparse_rows_into(*s.rows)
    r.topk_into(c["topk"], *s.top)
    steps = r.info().steps
    r.free()
    if kind == "job":
        G.free()
    return [steps, nnz, *s.rows, *s.top]


def work(case):
    """Each input once and each output once: the CSR (16 bytes a node's row
    and 8 an edge where the graph is loaded in the pass; where it is resident,
    no more of it than one 32-byte sector a draw), one id and one count for
    every stored pair and top-k place.  Integer operations of the draws
    (Philox4x32-10: about 60 a draw, two multiplications and three logical
    operations in each of ten rounds, and the search) stand in for flops."""
    kind, R, topk = case["kind"], case["R"], case["topk"]
    if case["graph"] == "rmat":
        n = 1 << case["scale"]
        m = 16 * n
    elif case["graph"] == "chunglu_batch":
        n = int(case["count"] * (case["nmax"] - case["nmin"]) / math.log(case["nmax"] / case["nmin"]))
        m = 12 * n
    else:
        n = case["n"]
        m = case.get("m", 12 * n)
    S = n
    if kind == "list":
        S = case["sources"]
    if kind == "range":
        S = n // case["part"]
    if kind == "serve":
        S = int(case["queries"] * (case["smax"] - 1) / math.log(max(2, case["smax"])))
    draws = S * R / case["alpha"]
    graph = 8.0 * n + 8.0 * m
    if kind not in ("job", "host"):
        graph = min(graph, 32.0 * draws)
    pairs = 0 if kind in ("list", "serve") else S * min(R, n) * 0.65  # distinct endpoints of a source, about
    return {"bytes": graph + 8.0 * pairs + 8.0 * S * topk, "flops": 60.0 * draws}


def exact(case, seed):
    """Every output is a whole number: compared bit by bit, no value in 64 bits stands beside it."""
    return None
