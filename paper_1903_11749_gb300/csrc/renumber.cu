// renumber.cu -- the walk layout's own node numbering.
//
// Nodes are numbered class by class (ClassTab in ppr_internal.cuh: dangling,
// single edge, degree, or the number of ranges 2^c of the row), because a
// node's place within its class is then all a walk needs to find its slots.
// Within a class they keep the caller's order.  (Descending in-degree order
// within the classes, which packs the rows most walks pass, was measured:
// R-MAT scale 24 walker 23.461 against 23.470 ms without it, alias 23.571
// against 23.587, scale 22 21.581 against 21.589; with a slot a draw there is
// no small hot record left to pack.)  The numbering is internal: sources,
// result rows and top-k use the caller's ids, and the draw of a walk is keyed
// by the caller's source id, so every count is the same under any numbering.
//   order[seq]: caller id (within its instance);  code_of[v]: code of caller node v.
#include "ppr_host.h"
#include "scan.cuh"

namespace ppr {

struct NumberArgs {
    int64_t n, m;
    const int64_t *row_ptr;
    uint32_t lam_bits;
    bool wide, exact;
    int64_t tiles;
    uint32_t tile;          // nodes a warp takes
    uint32_t *hist;         // [class][tile]
    uint64_t *off;          // its exclusive scan
    uint32_t *heads;        // bit e: a row starts at edge e
    LayoutStats *st;
    const int64_t *node_off;
    int32_t count;
    int32_t *order;
    uint32_t *code_of;
};

// Degree of caller row v, 0 (and a flag) when its row_ptr is invalid.
__device__ __forceinline__ uint32_t checked_degree(const NumberArgs &A, int64_t v, int64_t &a, uint32_t &flags)
{
    a = A.row_ptr[v];
    const int64_t b = A.row_ptr[v + 1];
    if (a < 0 || b < a || b > A.m || (v == 0 && a != 0) || (v == A.n - 1 && b != A.m)) {
        flags |= kBadRowPtr;
        return 0;
    }
    if (b - a > PPR_MAX_DEGREE) {
        flags |= kBigDegree;
        return 0;
    }
    return (uint32_t)(b - a);
}

__device__ __forceinline__ uint32_t node_class(const NumberArgs &A, uint32_t d)
{
    return class_of_degree(d, A.lam_bits, A.wide, A.exact);
}

// Per-tile class counts; row starts and degree statistics.  Four warps a
// block, one tile a warp.
__global__ void __launch_bounds__(128) k_rn_hist(NumberArgs A)
{
    __shared__ uint32_t h_all[4 * kClasses];
    const uint32_t wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
    uint32_t *h = h_all + wid * kClasses;
    const int64_t t = (int64_t)blockIdx.x * 4 + wid;
    for (uint32_t i = lane; i < kClasses; i += 32) h[i] = 0;
    __syncwarp();
    uint32_t dmax = 0, dang = 0, flags = 0;
    if (t < A.tiles) {
        for (uint32_t r = 0; r < A.tile; r += 32) {
            const int64_t v = t * A.tile + r + lane;
            uint32_t key = 0xffffffffu;
            if (v < A.n) {
                int64_t a;
                const uint32_t d = checked_degree(A, v, a, flags);
                dmax = max(dmax, d);
                dang += d == 0;
                key = node_class(A, d);
                if (d) atomicOr(&A.heads[a >> 5], 1u << (a & 31));
            }
            const uint32_t peers = __match_any_sync(0xffffffffu, key);
            if (v < A.n && lane == (uint32_t)(__ffs(peers) - 1)) h[key] += __popc(peers);
            __syncwarp();
        }
        for (uint32_t i = lane; i < kClasses; i += 32) A.hist[(int64_t)i * A.tiles + t] = h[i];
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        dmax = max(dmax, __shfl_xor_sync(0xffffffffu, dmax, o));
        dang += __shfl_xor_sync(0xffffffffu, dang, o);
        flags |= __shfl_xor_sync(0xffffffffu, flags, o);
    }
    if (lane == 0) {
        if (dmax) atomicMax(&A.st->max_degree, (unsigned long long)dmax);
        if (dang) atomicAdd(&A.st->dangling, (unsigned long long)dang);
        if (flags) atomicOr(&A.st->status, flags);
    }
}

// What the host needs to lay the classes out: the statistics and each class's first seq.
struct ClassStarts {
    LayoutStats st;
    uint64_t start[kClasses + 1];
};

__global__ void k_rn_starts(NumberArgs A, ClassStarts *out)
{
    const uint32_t i = threadIdx.x;
    if (i <= kClasses) out->start[i] = A.off[(int64_t)i * A.tiles];
    if (i == 0) out->st = *A.st;
}

struct ClassEntries {
    uint32_t e0[kClasses];  // first table entry of each class
    uint32_t start[kClasses];
};

// Stable scatter: node v of tile t goes to off[class][t] plus the number of
// earlier nodes of the tile in its class.
__global__ void __launch_bounds__(128) k_rn_scatter(NumberArgs A, ClassEntries C)
{
    __shared__ uint32_t seen_all[4 * kClasses];
    const uint32_t wid = threadIdx.x >> 5, lane = threadIdx.x & 31;
    uint32_t *seen = seen_all + wid * kClasses;
    const int64_t t = (int64_t)blockIdx.x * 4 + wid;
    for (uint32_t i = lane; i < kClasses; i += 32) seen[i] = 0;
    __syncwarp();
    if (t >= A.tiles) return;
    for (uint32_t r = 0; r < A.tile; r += 32) {
        const int64_t v = t * A.tile + r + lane;
        uint32_t key = 0xffffffffu;
        if (v < A.n) {
            int64_t a;
            uint32_t flags = 0;
            key = node_class(A, checked_degree(A, v, a, flags));
        }
        const uint32_t peers = __match_any_sync(0xffffffffu, key);
        const uint32_t before = __popc(peers & ((1u << lane) - 1));
        uint32_t base = 0;
        if (v < A.n) base = seen[key];
        __syncwarp();
        if (v < A.n) {
            const uint32_t seq = (uint32_t)A.off[(int64_t)key * A.tiles + t] + base + before, idx = seq - C.start[key];
            int64_t id = v;
            if (A.count > 0) {  // the id within its instance
                int32_t lo = 0, hi = A.count;
                while (hi - lo > 1) {
                    const int32_t mid = (lo + hi) >> 1;
                    if (A.node_off[mid] <= v) lo = mid;
                    else hi = mid;
                }
                id -= A.node_off[lo];
            }
            A.order[seq] = (int32_t)id;
            A.code_of[v] = ((C.e0[key] + (idx >> kIdxBits)) << kIdxBits) | (idx & kIdxMask);
            if (before == 0) seen[key] = base + __popc(peers);
        }
        __syncwarp();
    }
}

int number_nodes(const ppr_ctx *ctx, int64_t n, int64_t m, const int64_t *d_rp, const int64_t *d_off, uint32_t *heads,
                 LayoutStats *d_stats, bool wide, cudaStream_t st, ppr_graph *g, std::vector<void *> &tmp)
{
    Range range("number nodes");
    int rc;
    NumberArgs A{};
    A.n = n;
    A.m = m;
    A.row_ptr = d_rp;
    A.lam_bits = g->lam_bits;
    A.wide = wide;
    A.exact = g->instances == 0 && n <= kExactNodes && (ctx->force_exact < 0 ? n > kExactMin : ctx->force_exact == 1);
    // nodes a warp takes in turn: few where the graph is small (a warp's chain
    // of rounds is then the kernel's time)
    A.tile = n <= 2048 ? 32u : (n <= (1 << 18) ? 128u : 1024u);
    A.tiles = (n + A.tile - 1) / A.tile;
    A.heads = heads;
    A.st = d_stats;
    A.node_off = d_off;
    A.count = g->instances;
    A.order = g->order;
    A.code_of = g->code_of;
    const int64_t cells = A.tiles * kClasses;
    uint64_t *scan_tmp;
    ClassStarts *d_cs;
    if ((rc = dev_alloc((void **)&A.hist, sizeof(uint32_t) * cells, "class counts", st))) return rc;
    tmp.push_back(A.hist);
    if ((rc = dev_alloc((void **)&A.off, sizeof(uint64_t) * (cells + 1), "class offsets", st))) return rc;
    tmp.push_back(A.off);
    if ((rc = dev_alloc((void **)&scan_tmp, sizeof(uint64_t) * ((cells + kScanTile - 1) / kScanTile + 2), "scan scratch",
                        st)))
        return rc;
    tmp.push_back(scan_tmp);
    if ((rc = dev_alloc((void **)&d_cs, sizeof(ClassStarts), "class starts", st))) return rc;
    tmp.push_back(d_cs);
    const unsigned tb = (unsigned)((A.tiles + 3) / 4);
    k_rn_hist<<<tb, 128, 0, st>>>(A);
    note_launch();
    exclusive_scan_u32(A.hist, cells, A.off, scan_tmp, st);
    k_rn_starts<<<1, 64, 0, st>>>(A, d_cs);
    note_launch();
    ClassStarts cs;
    PPR_CUDA(cudaMemcpyAsync(&cs, d_cs, sizeof(cs), cudaMemcpyDeviceToHost, st));
    PPR_CUDA(cudaStreamSynchronize(st));
    if (cs.st.status & kBadRowPtr) {
        set_error("row_ptr must start at 0, be non-decreasing and end at m");
        return PPR_EINVAL;
    }
    if (cs.st.status & kBigDegree) {
        set_error("an out-degree exceeds the limit %lld", (long long)PPR_MAX_DEGREE);
        return PPR_ERANGE;
    }
    g->max_degree = (int64_t)cs.st.max_degree;
    g->dangling = (int64_t)cs.st.dangling;
    ClassEntries C{};
    ClassTab &T = g->htab;
    uint32_t e = 0;
    g->n_slots = g->n_single = 0;
    for (uint32_t c = 0; c < kClasses; ++c) {
        C.e0[c] = e;
        C.start[c] = (uint32_t)cs.start[c];
        for (uint64_t at = cs.start[c]; at < cs.start[c + 1]; at += 1ull << kIdxBits, ++e) {
            const uint64_t cnt = std::min<uint64_t>(cs.start[c + 1] - at, 1ull << kIdxBits);
            T.e[e] = TabEntry{0, kKindDangling, (uint32_t)at};
            g->degree[e] = c <= kExact ? c : 0;
            if (c == 1) {
                T.e[e].kind = kKindSingle;
                T.e[e].addr = sizeof(uint32_t) * (uint64_t)g->n_single;
                g->n_single += (int64_t)cnt;
            } else if (c >= 2) {
                // entries start on 32 slots, so that a warp of the slot build has one row where rows have 32 ranges
                g->n_slots = (g->n_slots + 31) & ~31ll;
                T.e[e].kind = c <= kExact ? ranges_log2(c, g->lam_bits, wide) : c - kExact - 1;
                T.e[e].addr = sizeof(Sector) * (uint64_t)g->n_slots;
                g->n_slots += (int64_t)(cnt << T.e[e].kind);
            }
        }
    }
    for (; e < kTabEntries; ++e) T.e[e] = TabEntry{0, kKindDangling, 0xffffffffu};
    k_rn_scatter<<<tb, 128, 0, st>>>(A, C);
    note_launch();
    PPR_CUDA(cudaGetLastError());
    return PPR_OK;
}

}  // namespace ppr
