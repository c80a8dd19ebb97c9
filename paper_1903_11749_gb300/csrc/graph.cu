// graph.cu -- device construction of the walk layout (edge records with
// per-row inclusive weight prefixes, guide slots) and of the depth-3 segment
// tables and the alias tables.
//
// Sec. 2.1 defines the routing probability r(s,t) = w(<s,t>) / sum_v w(<s,v>).
// The step rule realises it exactly over integers with the row's inclusive
// prefix P and total W_u: the next edge is the first e with P[e] > x for x
// uniform on [0, W_u).  Algorithm 4 ("big moves") precomputes, for small
// nodes, the distribution over short walk outcomes; here it is built with a
// fixed depth of 3 in 2^62 fixed point, one warp per node.
#include <cstdio>
#include <type_traits>

#include "ppr_host.h"
#include "scan.cuh"

namespace ppr {

// ------------------------------------------------------------ edge records ----
// Prefixes by edge, not by row: a scan of the weights that restarts at every
// row start (the bits number_nodes set) gives each edge its inclusive prefix
// P.  Every thread takes eight consecutive edges whatever the rows are, so a
// hub of a million edges and a million rows of one edge cost the same, where
// a build by rows needs a tier of kernels per row length and still waits for
// the longest row of each.  Two reads of the weights (tile sums, then the
// records), no tier lists, no host round trip between them.
constexpr uint32_t kEdgeThreads = 512, kEdgeRun = 8;
constexpr uint32_t kEdgeTile = kEdgeThreads * kEdgeRun;
constexpr uint32_t kSelfCarry = 512;  // up to so many tiles each block adds up the tiles before it itself

// Running sum since the last row start; bit 63: a row starts in the range.
using Run = unsigned long long;
constexpr Run kRowStart = 1ull << 63;
__device__ __forceinline__ Run run_join(Run a, Run b) { return (b & kRowStart) ? b : a + b; }

// Join of the runs of all threads before this one (threads in order); *total: of all.
__device__ __forceinline__ Run block_runs(Run v, Run *s_warp, Run *total)
{
    const uint32_t lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    Run x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const Run y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= (uint32_t)o) x = run_join(y, x);
    }
    Run before = __shfl_up_sync(0xffffffffu, x, 1);
    if (lane == 0) before = 0;
    if (lane == 31) s_warp[wid] = x;
    __syncthreads();
    Run carry = 0, all = 0;
    for (uint32_t q = 0; q < nw; ++q) {
        if (q == wid) carry = all;
        all = run_join(all, s_warp[q]);
    }
    __syncthreads();
    if (total) *total = all;
    return run_join(carry, before);
}

struct EdgeArgs {
    int64_t n, m;
    const int32_t *col;
    const uint32_t *w;
    const uint32_t *heads;
    const int64_t *row_ptr;
    const int64_t *node_off;  // batched graphs
    int32_t count;
    const uint32_t *code_of;
    Run *tile;                // per tile: its run, then (more than kSelfCarry tiles) the join of those before it
    int64_t tiles;
    void *edges;
    LayoutStats *st;
    bool vec;                 // col and w are 16-byte aligned
};

__device__ __forceinline__ void load8(const uint32_t *p, int64_t e0, int64_t m, bool vec, uint32_t (&v)[kEdgeRun])
{
    if (vec && e0 + kEdgeRun <= m) {
        const uint4 a = __ldg(reinterpret_cast<const uint4 *>(p + e0)), b = __ldg(reinterpret_cast<const uint4 *>(p + e0) + 1);
        v[0] = a.x, v[1] = a.y, v[2] = a.z, v[3] = a.w, v[4] = b.x, v[5] = b.y, v[6] = b.z, v[7] = b.w;
    } else {
#pragma unroll
        for (uint32_t i = 0; i < kEdgeRun; ++i) v[i] = e0 + i < m ? __ldg(p + e0 + i) : 0u;
    }
}

__device__ __forceinline__ uint32_t heads8(const EdgeArgs &A, int64_t e0)
{
    return e0 < A.m ? (A.heads[e0 >> 5] >> (e0 & 31)) & 0xffu : 0u;
}

__device__ __forceinline__ Run run8(const uint32_t (&w)[kEdgeRun], uint32_t hb)
{
    Run r = 0;
#pragma unroll
    for (uint32_t i = 0; i < kEdgeRun; ++i) r = ((hb >> i) & 1u) ? (kRowStart | w[i]) : r + w[i];
    return r;
}

__global__ void __launch_bounds__(kEdgeThreads) k_edge_tiles(EdgeArgs A)
{
    __shared__ Run s_warp[kEdgeThreads / 32];
    const int64_t e0 = ((int64_t)blockIdx.x * kEdgeThreads + threadIdx.x) * kEdgeRun;
    uint32_t w[kEdgeRun];
    load8(A.w, e0, A.m, A.vec, w);
    Run total;
    block_runs(run8(w, heads8(A, e0)), s_warp, &total);
    if (threadIdx.x == 0) A.tile[blockIdx.x] = total;
}

__global__ void __launch_bounds__(1024) k_edge_carry(EdgeArgs A)
{
    __shared__ Run s_warp[32];
    Run carry = 0;
    for (int64_t t0 = 0; t0 < A.tiles; t0 += 4 * 1024) {  // four consecutive tiles a thread
        Run v[4], mine = 0, all;
        const int64_t t = t0 + 4 * (int64_t)threadIdx.x;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            v[i] = t + i < A.tiles ? A.tile[t + i] : 0ull;
            mine = run_join(mine, v[i]);
        }
        Run before = run_join(carry, block_runs(mine, s_warp, &all));
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            if (t + i < A.tiles) A.tile[t + i] = before;
            before = run_join(before, v[i]);
        }
        carry = run_join(carry, all);
    }
}

template <bool WIDE>
__global__ void __launch_bounds__(kEdgeThreads) k_edge_records(EdgeArgs A)
{
    __shared__ Run s_warp[kEdgeThreads / 32];
    __shared__ uint32_t s_flags;
    if (threadIdx.x == 0) s_flags = 0;
    const int64_t e0 = ((int64_t)blockIdx.x * kEdgeThreads + threadIdx.x) * kEdgeRun;
    uint32_t w[kEdgeRun], c[kEdgeRun], flags = 0;
    load8(A.w, e0, A.m, A.vec, w);
    load8(reinterpret_cast<const uint32_t *>(A.col), e0, A.m, A.vec, c);
    // targets to codes: eight independent loads in flight
    int32_t g = 0;
    int64_t g_end = A.m, base = 0, size = A.n;  // the instance of the edge at hand
    if (A.count > 0 && e0 < A.m) {
        int32_t lo = 0, hi = A.count;
        while (hi - lo > 1) {  // last instance whose first edge is <= e0
            const int32_t mid = (lo + hi) >> 1;
            if (A.row_ptr[A.node_off[mid]] <= e0) lo = mid;
            else hi = mid;
        }
        g = lo;
        base = A.node_off[g];
        size = A.node_off[g + 1] - base;
        g_end = A.row_ptr[A.node_off[g + 1]];
    }
#pragma unroll
    for (uint32_t i = 0; i < kEdgeRun; ++i) {
        if (e0 + i < A.m) {
            if (A.count > 0)
                while (e0 + i >= g_end) {
                    ++g;
                    base = A.node_off[g];
                    size = A.node_off[g + 1] - base;
                    g_end = A.row_ptr[A.node_off[g + 1]];
                }
            if (w[i] == 0) flags |= kBadWeight;
            if ((int64_t)(int32_t)c[i] < 0 || (int64_t)(int32_t)c[i] >= size) flags |= kBadCol, c[i] = 0;
            else c[i] = __ldg(A.code_of + base + c[i]);
        }
    }
    const uint32_t hb = heads8(A, e0);
    Run before = block_runs(run8(w, hb), s_warp, nullptr);
    Run carry;
    if (A.tiles > kSelfCarry) {
        carry = A.tile[blockIdx.x];
    } else {  // the tiles before this one (up to one a thread)
        const Run v = threadIdx.x < blockIdx.x ? A.tile[threadIdx.x] : 0ull;
        block_runs(v, s_warp, &carry);
    }
    Run P = run_join(carry, before) & ~kRowStart;
    uint64_t v[kEdgeRun];
#pragma unroll
    for (uint32_t i = 0; i < kEdgeRun; ++i) {
        P = ((hb >> i) & 1u) ? (Run)w[i] : P + w[i];
        v[i] = P;
        if (!WIDE && P >= (1ull << 32)) flags |= kWide;
    }
    if (e0 < A.m) {  // (the array is padded to whole runs)
        if constexpr (WIDE) {
            Sector *dst = reinterpret_cast<Sector *>(static_cast<EdgeW *>(A.edges) + e0);
#pragma unroll
            for (uint32_t i = 0; i < kEdgeRun; i += 2)
                st_sector(dst + i / 2, Sector{{(uint32_t)v[i], (uint32_t)(v[i] >> 32), c[i], 0u, (uint32_t)v[i + 1],
                                               (uint32_t)(v[i + 1] >> 32), c[i + 1], 0u}});
        } else {
            Sector *dst = reinterpret_cast<Sector *>(static_cast<EdgeN *>(A.edges) + e0);
#pragma unroll
            for (uint32_t i = 0; i < kEdgeRun; i += 4)
                st_sector(dst + i / 4, Sector{{(uint32_t)v[i], c[i], (uint32_t)v[i + 1], c[i + 1], (uint32_t)v[i + 2],
                                               c[i + 2], (uint32_t)v[i + 3], c[i + 3]}});
        }
    }
    if (flags) atomicOr(&s_flags, flags);
    __syncthreads();
    if (threadIdx.x == 0 && s_flags) atomicOr(&A.st->status, s_flags);
}

// ------------------------------------------------------------ nodes, slots ----
struct SlotArgs {
    int64_t n;
    const int64_t *row_ptr;
    const uint32_t *code_of;
    const ClassTab *tab;
    NodeRec *node;
    Sector *slots;
    int64_t n_slots;
    const LayoutStats *st;
};

// Node records by seq, and the targets of single-edge nodes.
template <class E>
__global__ void __launch_bounds__(256) k_nodes(SlotArgs A, E edges)
{
    const int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (v >= A.n) return;
    const int64_t a = A.row_ptr[v];
    const uint32_t d = (uint32_t)(A.row_ptr[v + 1] - a), code = A.code_of[v];
    uint64_t total = 0;
    if (d) {
        const typename E::Rec last = edges.load(a + d - 1);
        total = d == 1 ? (uint64_t)E::target(last) : E::key(last);
        if (d == 1) reinterpret_cast<uint32_t *>(A.tab->e[code >> kIdxBits].addr)[code & kIdxMask] = E::target(last);
    }
    A.node[seq_of(*A.tab, code)] = NodeRec{pack_word0((uint64_t)a, d), total};
}

// Index of the first edge of a row whose prefix exceeds x, among its n edges
// from lo on (there is one).  P: uint32_t (narrow) or uint64_t.
template <class E, class P>
__device__ __forceinline__ uint32_t first_above(const typename E::Edge *row, uint32_t lo, uint32_t n, P x)
{
    while (n > 1) {
        const uint32_t half = n >> 1;
        const bool below = __ldg(&row[lo + half - 1].P) <= x;
        lo += below ? half : 0u;
        n = below ? n - half : half;
    }
    return lo;
}

// The same for 32 ascending x, one a lane, all 32 lanes taking part: a 32-ary
// search for lane 0's edge (two or three dependent loads where bisection takes
// ten), then the edges from there on, 32 at a time in one load, each lane
// finding its place among them by shuffles.  A warp's ranges meet 16 to 64
// edges on average; after kWarpChunks loads (runs of light edges) the lanes left
// bisect what follows.
constexpr uint32_t kWarpChunks = 8;
template <class E, class P>
__device__ __forceinline__ uint32_t first_above_warp(const typename E::Edge *row, uint32_t d, P x)
{
    const uint32_t lane = threadIdx.x & 31;
    const P x0 = __shfl_sync(0xffffffffu, x, 0);
    uint32_t lo = 0, n = d;
    while (n > 32) {  // 32 parts; part i ends at edge lo + (i + 1) n / 32 - 1, the last one with P > x0
        const uint32_t end = lo + (uint32_t)(((uint64_t)(lane + 1) * n) >> 5) - 1;
        const uint32_t f = __popc(__ballot_sync(0xffffffffu, __ldg(&row[end].P) <= x0));
        const uint32_t a = (uint32_t)(((uint64_t)f * n) >> 5), b = (uint32_t)(((uint64_t)(f + 1) * n) >> 5);
        lo += a;
        n = b - a;
    }
    uint32_t at = 0;
    bool found = false;
    for (uint32_t chunk = 0; chunk < kWarpChunks; ++chunk, lo += 32) {
        const P v = lo + lane < d ? __ldg(&row[lo + lane].P) : (P)~(P)0;
        uint32_t cnt = 0;  // edges of the chunk with P <= x (31 at most where the last one is above x)
#pragma unroll
        for (uint32_t s = 16; s > 0; s >>= 1) cnt += __shfl_sync(0xffffffffu, v, cnt + s - 1) <= x ? s : 0u;
        const P last = __shfl_sync(0xffffffffu, v, 31);  // (by every lane, also those done)
        if (!found && last > x) {
            at = lo + cnt;
            found = true;
        }
        if (__all_sync(0xffffffffu, found)) break;
    }
    if (!found) at = first_above<E, P>(row, lo, d - lo, x);
    return at;
}

// One slot a thread.  The class-major numbering makes the slot's row and
// range plain arithmetic, neighbouring threads hold neighbouring ranges of a
// row, and every slot is one 32-byte store.  Bound by the latency of the
// searches: where a warp has 32 ranges of one row they search together
// (R-MAT scale 24, 394 M slots: 7.2 -> 5.3 ms; 64-bit keys and a table search a
// thread before that: 7.9).
template <class E>
__global__ void __launch_bounds__(256) k_slots(SlotArgs A, E edges)
{
    using P = typename std::conditional<E::kWide, uint64_t, uint32_t>::type;
    __shared__ ClassTab tab;
    __shared__ uint32_t s_entry;
    // an input that failed its checks (weights of 0, totals beyond 32 bits)
    // has no ascending prefixes to search; the host reports it
    if (A.st->status) return;
    if (threadIdx.x == 0) s_entry = 0;
    for (uint32_t i = threadIdx.x; i < kTabEntries; i += blockDim.x) tab.e[i] = A.tab->e[i];
    __syncthreads();
    // the last entry whose slots start at or before the block's first
    const uint64_t at0 = reinterpret_cast<uint64_t>(A.slots + (int64_t)blockIdx.x * blockDim.x);
    if (threadIdx.x < kTabEntries && tab.e[threadIdx.x].kind < kKindSingle && tab.e[threadIdx.x].addr <= at0)
        atomicMax(&s_entry, threadIdx.x);
    __syncthreads();
    const int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= A.n_slots) return;
    const uint64_t at = reinterpret_cast<uint64_t>(A.slots + s);
    uint32_t entry = s_entry;  // slot entries follow each other in the table
    while (entry + 1 < kTabEntries && tab.e[entry + 1].kind < kKindSingle && tab.e[entry + 1].addr <= at) ++entry;
    const TabEntry t = tab.e[entry];
    const uint32_t c = t.kind, rel = (uint32_t)((at - t.addr) / sizeof(Sector));  // below 2^32: a device holds fewer slots
    const uint32_t b = rel & ((1u << c) - 1);
    // slots between the entry's last row and the next entry's start belong to no row (whole warps where c >= 5)
    const uint32_t next = entry + 1 < kTabEntries ? tab.e[entry + 1].first : 0xffffffffu;
    if (t.first + (rel >> c) >= (next == 0xffffffffu ? (uint32_t)A.n : next)) return;
    const NodeRec r = A.node[t.first + (rel >> c)];
    const typename E::Edge *row = edges.e + (r.word0 & kBeginMask);
    const uint32_t d = (uint32_t)(r.word0 >> 40) & kCountMask;
    const uint64_t W = r.total;
    P X0, X1;  // the range's first x and its last: ceil((b + 1) W / 2^c) - 1
    if constexpr (E::kWide) {
        X0 = range_start(W, b, c);
        X1 = range_start(W, b + 1, c) - (((W * (b + 1ull)) & ((1ull << c) - 1)) == 0);
    } else {
        const uint64_t lo = (uint64_t)(uint32_t)W * b, up = lo + (uint32_t)W;
        X0 = (uint32_t)(lo >> c);
        X1 = (uint32_t)(up >> c) - (((uint32_t)up & ((1u << c) - 1)) == 0);
    }
    uint32_t lo = 0;
    if (c >= 5) lo = first_above_warp<E, P>(row, d, X0);
    else if (c) lo = first_above<E, P>(row, 0, d, X0);
    const uint32_t left = d - lo;  // edges from lo to the row's end
    constexpr uint32_t kFit = E::kWide ? 3 : 4;
    typename E::Rec rec[kFit];
    uint32_t q = 0;  // edges that meet the range, 0 for more than fit
#pragma unroll
    for (uint32_t i = 0; i < kFit; ++i) rec[i] = __ldg(reinterpret_cast<const typename E::Rec *>(row) + lo + min(i, left - 1));
#pragma unroll
    for (uint32_t i = 0; i < kFit; ++i)
        if (q == 0 && (P)E::key(rec[i]) > X1) q = i + 1;
    const uint64_t e_lo = (r.word0 & kBeginMask) + lo;
    Sector o;
#pragma unroll
    for (int i = 0; i < 8; ++i) o.v[i] = 0;
    o.v[0] = (uint32_t)W;
    if constexpr (!E::kWide) {
        if (q) {
#pragma unroll
            for (uint32_t i = 0; i < 3; ++i) o.v[1 + i] = i + 1 < q ? rec[i].x : 0xffffffffu;
            uint32_t to = E::target(rec[0]);
#pragma unroll
            for (uint32_t i = 0; i < 4; ++i) {
                if (i < q) to = E::target(rec[i]);
                o.v[4 + i] = to;
            }
        } else {
            const uint64_t e_hi = (r.word0 & kBeginMask) + first_above<E, P>(row, lo + kFit, left - kFit, X1), sec = e_lo >> 2;
            const uint32_t nsec = (uint32_t)((e_hi >> 2) - sec + 1), gs = (nsec + kGroups - 1) / kGroups;
            uint32_t k[kGroups - 1];
#pragma unroll
            for (uint32_t g = 0; g < kGroups - 1; ++g)
                k[g] = (g + 1) * gs < nsec ? __ldg(&edges.e[4 * (sec + (uint64_t)(g + 1) * gs) - 1].P) : 0xffffffffu;
            o.v[1] = k[0];
            o.v[2] = k[1];
            o.v[3] = k[2];
            o.v[7] = k[3];
            o.v[4] = kMarkOverflow | ((uint32_t)(e_lo & 3) << 8) | (uint32_t)(sec >> 32);
            o.v[5] = (uint32_t)sec;
            o.v[6] = nsec;
        }
    } else {
        o.v[1] = (uint32_t)(W >> 32);
        if (q && X1 - X0 < (1ull << 32)) {
#pragma unroll
            for (uint32_t i = 0; i < 2; ++i) o.v[2 + i] = i + 1 < q ? (uint32_t)(E::key(rec[i]) - X0) : 0xffffffffu;
            uint32_t to = E::target(rec[0]);
#pragma unroll
            for (uint32_t i = 0; i < 3; ++i) {
                if (i < q) to = E::target(rec[i]);
                o.v[4 + i] = to;
            }
        } else {
            const uint32_t hi = q ? lo + q - 1 : first_above<E, P>(row, lo + kFit, left - kFit, X1);
            o.v[4] = kMarkOverflow;
            o.v[5] = (uint32_t)e_lo;
            o.v[6] = (uint32_t)(e_lo >> 32);
            o.v[7] = hi - lo + 1;
        }
    }
    st_sector(A.slots + s, o);
}

// The layout of CSR (d_rp, d_col, d_w).  Returns PPR_OK, an error, or 1 when
// a row total reaches 2^32 and WIDE is false (the caller then builds the wide
// layout).
template <class E>
static int build_layout(ppr_ctx *ctx, int64_t n, int64_t m, const int64_t *d_rp, const int32_t *d_col,
                        const uint32_t *d_w, const int64_t *d_off, cudaStream_t st, ppr_graph *g,
                        std::vector<void *> &tmp)
{
    int rc;
    // Ranges per row: at most 2^lam_bits edges a range on average.  One edge a
    // range makes overflow rare (5 % of the draws with Zipf weights, 11 % with
    // two), two halve the slots (45 and 23 bytes an edge).  What decides is
    // where the slots lie: within L2 the second load of an overflow costs
    // more, far beyond it (16 times) every slot is a miss anyway and the
    // overflow one more; in between the smaller slots hit L2 more often.
    // Walker ms with one / two: R-MAT scale 16 .347 / .375, 18 1.22 / 1.29, 19
    // 2.70 / 2.52, 20 6.12 / 5.82, 22 7.42 / 7.76 (2^20 sources), 24 86.2 /
    // 91.5; Chung-Lu 2.4 M edges .724 / .777, 12 M 5.45 / 4.37.  A batch's
    // instances are walked one after the other: the largest counts (256
    // graphs: 17.6 / 19.0).  The wide layout's slot holds three edges, and
    // its ranges one.  Slots that would take more than an eighth of the
    // device (64 m >> lam_bits bytes at most) get longer ranges.
    double share = 1.0;
    if (g->instances > 0) {
        int64_t largest = 0;
        for (int32_t i = 0; i < g->instances; ++i) largest = std::max(largest, g->node_off[i + 1] - g->node_off[i]);
        share = (double)largest / (double)n;
    }
    const double slot_bytes = 45.0 * (double)m * share, l2 = (double)ctx->l2_bytes;
    g->lam_bits = !E::kWide && slot_bytes > 1.75 * l2 && slot_bytes < 16.0 * l2 ? 1 : 0;
    while (g->lam_bits < 23 && (uint64_t)m * 64 >> g->lam_bits > ctx->mem_bytes / 8) ++g->lam_bits;
    if (ctx->force_lam >= 0) g->lam_bits = (uint32_t)ctx->force_lam;
    uint32_t *heads;
    LayoutStats *d_ls;
    const int64_t tiles = (m + kEdgeTile - 1) / kEdgeTile;
    const size_t head_words = (size_t)(m / 32 + 1);
    if ((rc = dev_alloc((void **)&heads, sizeof(uint32_t) * head_words, "row starts", st))) return rc;
    tmp.push_back(heads);
    if ((rc = dev_alloc((void **)&d_ls, sizeof(LayoutStats), "layout stats", st))) return rc;
    tmp.push_back(d_ls);
    Run *d_tile;
    if ((rc = dev_alloc((void **)&d_tile, sizeof(Run) * (tiles > 0 ? tiles : 1), "weight sums", st))) return rc;
    tmp.push_back(d_tile);
    if ((rc = dev_alloc((void **)&g->order, sizeof(int32_t) * n, "node order", st)) ||
        (rc = dev_alloc((void **)&g->code_of, sizeof(uint32_t) * n, "node codes", st)))
        return rc;
    PPR_CUDA(cudaMemsetAsync(heads, 0, sizeof(uint32_t) * head_words, st));
    PPR_CUDA(cudaMemsetAsync(d_ls, 0, sizeof(LayoutStats), st));
    if ((rc = number_nodes(ctx, n, m, d_rp, d_off, heads, d_ls, E::kWide, st, g, tmp))) return rc;
    const size_t run = kEdgeRun * sizeof(typename E::Edge);
    const size_t edge_bytes = (size_t)(tiles > 0 ? (m + kEdgeRun - 1) / kEdgeRun : 1) * run;
    if ((rc = dev_alloc(&g->edges, edge_bytes, "edge records", st)) ||
        (rc = dev_alloc((void **)&g->node, sizeof(NodeRec) * n, "node records", st)) ||
        (rc = dev_alloc((void **)&g->slots, sizeof(Sector) * std::max<int64_t>(g->n_slots, 1), "guide slots", st)) ||
        (rc = dev_alloc((void **)&g->single, sizeof(uint64_t) * (g->n_single / 2 + 1), "single targets", st)) ||
        (rc = dev_alloc((void **)&g->tab, sizeof(ClassTab), "class table", st)))
        return rc;
    for (TabEntry &t : g->htab.e) {
        if (t.kind < kKindSingle) t.addr += reinterpret_cast<uint64_t>(g->slots);
        if (t.kind == kKindSingle) t.addr += reinterpret_cast<uint64_t>(g->single);
    }
    PPR_CUDA(cudaMemcpyAsync(g->tab, &g->htab, sizeof(ClassTab), cudaMemcpyHostToDevice, st));
    g->device_bytes = (int64_t)(edge_bytes + (sizeof(NodeRec) + 8) * n + sizeof(Sector) * g->n_slots + 4 * g->n_single);
    EdgeArgs A{n, m, d_col, d_w, heads, d_rp, d_off, g->instances, g->code_of, d_tile, tiles, g->edges, d_ls,
               ((reinterpret_cast<uintptr_t>(d_col) | reinterpret_cast<uintptr_t>(d_w)) & 15) == 0};
    if (tiles > 0) {
        if (tiles > 1) {
            k_edge_tiles<<<(unsigned)tiles, kEdgeThreads, 0, st>>>(A);
            note_launch();
        }
        if (tiles > kSelfCarry) {
            k_edge_carry<<<1, 1024, 0, st>>>(A);
            note_launch();
        }
        k_edge_records<E::kWide><<<(unsigned)tiles, kEdgeThreads, 0, st>>>(A);
        note_launch();
    }
    const E edges{static_cast<const typename E::Edge *>(g->edges)};
    const SlotArgs B{n, d_rp, g->code_of, g->tab, g->node, g->slots, g->n_slots, d_ls};
    k_nodes<E><<<(unsigned)((n + 255) / 256), 256, 0, st>>>(B, edges);
    note_launch();
    if (g->n_slots > 0) {
        k_slots<E><<<(unsigned)((g->n_slots + 255) / 256), 256, 0, st>>>(B, edges);
        note_launch();
    }
    LayoutStats hs;
    PPR_CUDA(cudaGetLastError());
    PPR_CUDA(cudaMemcpyAsync(&hs, d_ls, sizeof(hs), cudaMemcpyDeviceToHost, st));
    PPR_CUDA(cudaStreamSynchronize(st));
    if (hs.status & kBadCol) {
        set_error("an edge target is outside [0, n) (of its instance)");
        return PPR_EINVAL;
    }
    if (hs.status & kBadWeight) {
        set_error("edge weights must be >= 1 (w(e) > 0, Sec. 2.1)");
        return PPR_EINVAL;
    }
    return (hs.status & kWide) ? 1 : PPR_OK;
}

int build_graph(ppr_ctx *ctx, int64_t n, int64_t m, const int64_t *row_ptr, const int32_t *col,
                const uint32_t *w, bool device_ptrs, bool renumber, cudaStream_t st, ppr_graph *g)
{
    const int64_t *d_rp = row_ptr;
    const int32_t *d_col = col;
    const uint32_t *d_w = w;
    std::vector<void *> tmp;
    auto cleanup = [&]() {
        for (void *p : tmp) dev_free(p, st);
        tmp.clear();
    };
    int rc;
    if (!device_ptrs) {
        void *p;
        if ((rc = dev_alloc(&p, sizeof(int64_t) * (n + 1), "row_ptr copy", st))) return cleanup(), rc;
        tmp.push_back(p);
        d_rp = (const int64_t *)p;
        if (m > 0) {
            if ((rc = dev_alloc(&p, sizeof(int32_t) * m, "col copy", st))) return cleanup(), rc;
            tmp.push_back(p);
            d_col = (const int32_t *)p;
            if ((rc = dev_alloc(&p, sizeof(uint32_t) * m, "w copy", st))) return cleanup(), rc;
            tmp.push_back(p);
            d_w = (const uint32_t *)p;
        }
        cudaError_t e = cudaMemcpyAsync((void *)d_rp, row_ptr, sizeof(int64_t) * (n + 1), cudaMemcpyHostToDevice, st);
        if (e == cudaSuccess && m > 0)
            e = cudaMemcpyAsync((void *)d_col, col, sizeof(int32_t) * m, cudaMemcpyHostToDevice, st);
        if (e == cudaSuccess && m > 0)
            e = cudaMemcpyAsync((void *)d_w, w, sizeof(uint32_t) * m, cudaMemcpyHostToDevice, st);
        if (e != cudaSuccess) return cleanup(), cuda_fail(e, "graph upload");
    }
    int64_t *d_off = nullptr;
    if (g->instances > 0) {  // kept with the graph: the walker reads instance offsets
        if ((rc = dev_alloc((void **)&g->d_node_off, sizeof(int64_t) * (g->instances + 1), "node_off", st)))
            return cleanup(), rc;
        d_off = g->d_node_off;
        cudaError_t e = cudaMemcpyAsync(d_off, g->node_off.data(), sizeof(int64_t) * (g->instances + 1),
                                        cudaMemcpyHostToDevice, st);
        if (e != cudaSuccess) return cleanup(), cuda_fail(e, "node_off upload");
    }
    rc = build_layout<NarrowEdges>(ctx, n, m, d_rp, d_col, d_w, d_off, st, g, tmp);
    g->renumbered = renumber && g->instances == 0;
    if (rc == 1) {  // some row total reaches 2^32: 64-bit prefixes
        for (void *p : {(void *)g->edges, (void *)g->node, (void *)g->slots, (void *)g->single, (void *)g->tab,
                        (void *)g->order, (void *)g->code_of})
            dev_free(p, st);
        g->edges = nullptr;
        g->node = nullptr;
        g->slots = nullptr;
        g->single = nullptr;
        g->tab = nullptr;
        g->order = nullptr;
        g->code_of = nullptr;
        g->wide = true;
        g->renumbered = false;
        rc = build_layout<WideEdges>(ctx, n, m, d_rp, d_col, d_w, d_off, st, g, tmp);
    }
    cleanup();
    return rc;
}

// ------------------------------------------------------------ segments ----

constexpr int kSegMaxDeg = 8;
constexpr int kSegMaxOut = 64;

__device__ __forceinline__ uint64_t mul_shift32(uint64_t q, uint32_t f)
{
    // floor(q * f / 2^32), q < 2^63
    uint64_t lo = q * (uint64_t)f;
    uint64_t hi = __umul64hi(q, (uint64_t)f);
    return (hi << 32) | (lo >> 32);
}

__device__ __forceinline__ uint64_t mul_div(uint64_t q, uint64_t num, uint64_t den)
{
    unsigned __int128 p = (unsigned __int128)q * num;
    return (uint64_t)(p / den);
}

// The layout's rows by seq, targets given by seq.
template <class E>
struct RowView {
    const NodeRec *node;
    E edges;
    const ClassTab *tab;
    __device__ __forceinline__ uint32_t deg(uint32_t u) const { return (uint32_t)(node[u].word0 >> 40) & kCountMask; }
    __device__ __forceinline__ uint64_t begin(uint32_t u) const { return node[u].word0 & kBeginMask; }
    // (the record of a single-edge row holds its target instead of its total)
    __device__ __forceinline__ uint64_t total(uint32_t u) const
    {
        uint32_t d = deg(u);
        if (d == 1) return 1;  // with wt = 1 above: the single edge has ratio 1
        return d ? node[u].total : 0ull;
    }
    // weight and target of the i-th edge of u
    __device__ __forceinline__ void edge(uint32_t u, uint32_t i, uint64_t &wt, uint32_t &tgt) const
    {
        const uint32_t d = deg(u);
        if (d == 1) {  // target kept in the node record; weight ratio is 1
            wt = 1;
            tgt = seq_of(*tab, (uint32_t)node[u].total);
            return;
        }
        uint64_t b = begin(u);
        auto r = edges.load(b + i);
        uint64_t prev = i > 0 ? E::key(edges.load(b + i - 1)) : 0ull;
        wt = E::key(r) - prev;
        tgt = seq_of(*tab, E::target(r));
    }
};

// Table entry of node seq v (entries are in seq order, unused ones last).
__device__ __forceinline__ uint32_t entry_of(const ClassTab &t, uint32_t v)
{
    uint32_t lo = 0, hi = kTabEntries;
    while (hi - lo > 1) {
        const uint32_t mid = (lo + hi) >> 1;
        if (t.e[mid].first <= v) lo = mid;
        else hi = mid;
    }
    return lo;
}

__device__ __forceinline__ uint32_t code_of_seq(const ClassTab &t, uint32_t v)
{
    const uint32_t e = entry_of(t, v);
    return (e << kIdxBits) | (v - t.e[e].first);
}

// Where a segment table is hung: the small classes' slots and single targets
// of the segment layout (copies of the plain layout's), see SegCache.
struct SegLinks {
    ClassTab *tab;
    uint32_t *single;
    SegHead *head;
};

// Segment tables in two passes.  k_seg_scan (every node; a warp takes 32 at a
// time) tests the
// depth-1 shape of all 32 nodes at once (degree <= 8 of the node and of its
// targets), then for each candidate left the depth-2 shape, and counts the
// raw contributions the path enumeration will make; eligible nodes are listed
// by that count (one reservation per warp and tier), with min(raw, 64)
// entries each, whose scan gives every listed node a fixed slot range.
// k_seg_fill (one warp per listed node) enumerates the paths once, level by
// level, sums equal outcomes in a shared-memory hash table, drops zero
// masses, rejects a node with more than 64 outcomes, puts the rest in
// canonical order (terminated before active, then node, then length) by
// ranking, and writes the table at the node's slot.  A table's place in the
// entry array is free (its link holds begin and count; a shorter table
// leaves a gap), so only its content is fixed.

constexpr unsigned long long kSegEmpty = ~0ull;  // free hash slot (an outcome key's node field is below 2^31)
constexpr uint32_t kSegSmallRaw = 128;  // raw contributions up to which the small table (256 slots) serves
constexpr int kSegLargeSlots = 2048;    // the largest raw count is 8 * (1 + 8 * (1 + 2 * 8)) = 1,096

struct SegCounters {
    unsigned int listed[2];       // nodes listed: [0] small table, [1] large table
    unsigned long long bound;     // sum over listed nodes of min(raw, 64): entries to allocate
    unsigned long long used;      // entries written
    unsigned long long tables;    // nodes given a table
};

// Path enumeration by level: depth-1 targets, then the pairs (i1, i2).
struct SegStage {
    unsigned long long s1_q[kSegMaxDeg], s1_W[kSegMaxDeg];
    unsigned long long s2_q[kSegMaxDeg * kSegMaxDeg], s2_W[kSegMaxDeg * kSegMaxDeg];
    uint32_t s1_node[kSegMaxDeg], s1_deg[kSegMaxDeg];
    uint32_t s2_node[kSegMaxDeg * kSegMaxDeg], s2_deg[kSegMaxDeg * kSegMaxDeg], s2_pre[kSegMaxDeg * kSegMaxDeg + 1];
};

// Compacted, then ranked outcomes; so: the keys with the caller's node ids
// (ranking on a renumbered layout).
struct SegRank {
    unsigned long long sk[kSegMaxOut], sq[kSegMaxOut], so[kSegMaxOut];
};

// Hash table of one warp: more slots than the tier's largest raw count, so it never fills.
template <int SLOTS>
struct SegHash {
    unsigned long long key[SLOTS];
    unsigned long long val[SLOTS];
    uint16_t used[SLOTS];          // claimed slots, in claim order
    union {  // one node at a time: the enumeration's staging, then the ranking's outcomes
        SegStage e;
        SegRank r;
    } u;
    unsigned int count;
    unsigned int full;  // a probe found no slot (cannot happen when the scan's count is right): no table
};

// list: listed nodes, small tier from the front, large from the back;
// lbound[list position]: min(raw contributions, 64), the entries the node's
// table may take (its slot range in the entry array comes from a scan of these).
template <class E>
__global__ void __launch_bounds__(256) k_seg_scan(RowView<E> G, int64_t n, uint32_t *list, uint32_t *lbound,
                                                  SegCounters *ct)
{
    const uint32_t lane = threadIdx.x & 31;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    // each warp takes 32 consecutive nodes (coalesced records, degree
    // test), then examines the candidates among them one by one with all lanes
    for (int64_t base = (int64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31u); base < n; base += stride) {
        const int64_t vl = base + lane;
        uint32_t dl = 0;
        bool c = false;
        if (vl < n) {
            const NodeRec r = G.node[vl];
            dl = (uint32_t)(r.word0 >> 40) & kCountMask;
            // depth 1, every lane its own node at once (most candidates have
            // a neighbour above the limit): the row's targets, then their degrees
            c = dl >= 1 && dl <= (uint32_t)kSegMaxDeg;
            if (c) {
                uint32_t tg[kSegMaxDeg];
                const uint64_t eb = r.word0 & kBeginMask;
#pragma unroll
                for (uint32_t i = 0; i < (uint32_t)kSegMaxDeg; ++i)
                    tg[i] = i >= dl ? 0u : seq_of(*G.tab, dl == 1 ? (uint32_t)r.total : E::target(G.edges.load(eb + i)));
#pragma unroll
                for (uint32_t i = 0; i < (uint32_t)kSegMaxDeg; ++i)
                    if (i < dl && G.deg(tg[i]) > (uint32_t)kSegMaxDeg) c = false;
            }
        }
        uint32_t cand = __ballot_sync(0xffffffffu, c);
        uint32_t listed_mask[2] = {0u, 0u}, my_bound = 0;  // this group's listed nodes (lane = node), per tier
        while (cand) {
            const uint32_t src_lane = __ffs(cand) - 1;
            cand &= cand - 1;
            const uint32_t v = (uint32_t)(base + src_lane);
            const uint32_t d1 = __shfl_sync(0xffffffffu, dl, src_lane);
            bool ok = true;
            uint32_t raw = 0;
            for (uint32_t p = lane; p < d1 * kSegMaxDeg; p += 32) {
                const uint32_t i1 = p / kSegMaxDeg, i2 = p % kSegMaxDeg;
                uint64_t wt;
                uint32_t a;
                G.edge(v, i1, wt, a);
                const uint32_t da = G.deg(a);
                if (da > (uint32_t)kSegMaxDeg) {
                    ok = false;
                    continue;
                }
                if (i2 == 0) raw += 1 + (da == 0);  // (a, terminated), and (a, active, 1) at a dead end
                if (i2 < da) {
                    uint32_t b;
                    G.edge(a, i2, wt, b);
                    const uint32_t db = G.deg(b);
                    if (db > (uint32_t)kSegMaxDeg) ok = false;
                    else raw += 1 + (db == 0) + 2 * db;  // (b, terminated), dead end, both outcomes at each c
                }
            }
            if (!__all_sync(0xffffffffu, ok)) continue;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) raw += __shfl_xor_sync(0xffffffffu, raw, o);
            listed_mask[raw <= kSegSmallRaw ? 0 : 1] |= 1u << src_lane;
            if (lane == src_lane) my_bound = min(raw, (uint32_t)kSegMaxOut);
        }
        // one reservation per tier for the group's listed nodes (not one
        // atomic per node: every warp would queue on the same counters)
        uint32_t res[2] = {0u, 0u};
        unsigned long long bsum = my_bound;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) bsum += __shfl_xor_sync(0xffffffffu, bsum, o);
        if (lane == 0) {
            if (listed_mask[0]) res[0] = atomicAdd(&ct->listed[0], (uint32_t)__popc(listed_mask[0]));
            if (listed_mask[1]) res[1] = atomicAdd(&ct->listed[1], (uint32_t)__popc(listed_mask[1]));
            if (bsum) atomicAdd(&ct->bound, bsum);
        }
        res[0] = __shfl_sync(0xffffffffu, res[0], 0);
        res[1] = __shfl_sync(0xffffffffu, res[1], 0);
#pragma unroll
        for (int tier = 0; tier < 2; ++tier) {
            if ((listed_mask[tier] >> lane) & 1u) {
                const uint32_t k = res[tier] + __popc(listed_mask[tier] & ((1u << lane) - 1));
                const int64_t pos = tier ? n - 1 - k : k;  // small tier from the front, large from the back
                list[pos] = (uint32_t)vl;
                lbound[pos] = my_bound;
            }
        }
    }
}

template <int SLOTS>
__device__ __forceinline__ void seg_insert(SegHash<SLOTS> *h, uint32_t node, uint32_t active, uint32_t len, uint64_t q)
{
    const unsigned long long key = ((unsigned long long)active << 63) | ((unsigned long long)node << 8) | len;
    uint32_t s = (node * 0x9E3779B1u ^ (len << 29) ^ (active << 31)) & (SLOTS - 1);
    for (uint32_t probe = 0; probe < (uint32_t)SLOTS; ++probe) {
        const unsigned long long prev = atomicCAS(&h->key[s], kSegEmpty, key);
        if (prev == kSegEmpty) h->used[atomicAdd(&h->count, 1u)] = (uint16_t)s;  // each claim takes a new slot
        if (prev == kSegEmpty || prev == key) {
            atomicAdd(&h->val[s], (unsigned long long)q);
            return;
        }
        s = (s + 1) & (SLOTS - 1);
    }
    h->full = 1;
}

// Tables of the nodes of one tier of `list`; SLOTS is above the tier's
// largest raw count.  Each warp's hash table is cleared once and restored
// slot by slot after each node.
// An outcome key with its node field replaced by the caller's id of that node.
__device__ __forceinline__ unsigned long long seg_key_caller(unsigned long long k, const int32_t *order)
{
    const uint32_t node = (uint32_t)((k >> 8) & 0x7fffffffull);
    return (k & ~(0x7fffffffull << 8)) | ((unsigned long long)(uint32_t)order[node] << 8);
}

// order: the layout's order array (the canonical order ranks outcomes by the
// caller's node ids).
// slot: first entry of the table of list position pos (exclusive scan of
// lbound), so a table is written without a shared counter.
template <class E, int SLOTS, int WARPS>
__global__ void __launch_bounds__(32 * WARPS) k_seg_fill(RowView<E> G, uint32_t T, const uint32_t *list, int tier,
                                                         int64_t n, SegCounters *ct, SegEntry *ent, SegLinks links,
                                                         const int32_t *order, const uint64_t *slot)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    SegHash<SLOTS> *h = reinterpret_cast<SegHash<SLOTS> *>(smem_raw) + (threadIdx.x >> 5);
    const uint32_t lane = threadIdx.x & 31, below = (1u << lane) - 1;
    for (uint32_t i = lane; i < (uint32_t)SLOTS; i += 32) {
        h->key[i] = kSegEmpty;
        h->val[i] = 0;
    }
    if (lane == 0) {
        h->count = 0;
        h->full = 0;
    }
    __syncwarp();
    const uint32_t listed = ct->listed[tier];
    const uint32_t cont = (uint32_t)(0x100000000ull - T);  // 2^32 - T, T >= 1
    const int64_t warps = (int64_t)gridDim.x * WARPS;
    unsigned long long w_used = 0, w_tables = 0;  // this warp's tables and their entries
    for (int64_t t = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; t < listed; t += warps) {
        const uint32_t v = list[tier ? n - 1 - t : t];
        const uint32_t d1 = G.deg(v);
        const uint64_t Wv = G.total(v);
        // all paths of length 1, 2, 3, level by level (the paper's masses in
        // 2^62 fixed point, the same arithmetic as the oracle's): the d1 edges
        // of v, then the pairs (i1, i2), then the triples, each level's
        // targets, masses and row totals staged in shared memory so that a
        // level costs one round of dependent loads for all its paths
        if (lane < d1) {
            uint64_t w1;
            uint32_t a;
            G.edge(v, lane, w1, a);
            const uint64_t q1 = mul_div(1ull << 62, w1, Wv);
            const uint32_t da = G.deg(a);
            seg_insert(h, a, 0, 0, mul_shift32(q1, T));
            if (da == 0) seg_insert(h, a, 1, 1, mul_shift32(q1, cont));
            h->u.e.s1_node[lane] = a;
            h->u.e.s1_deg[lane] = da;
            h->u.e.s1_q[lane] = mul_shift32(q1, cont);  // the mass that continues past a
            h->u.e.s1_W[lane] = da ? G.total(a) : 1ull;
        }
        __syncwarp();
        const uint32_t np = d1 * kSegMaxDeg;  // pair slots (i1, i2), i2 < deg(a_i1) valid
        for (uint32_t p = lane; p < np; p += 32) {
            const uint32_t i1 = p / kSegMaxDeg, i2 = p % kSegMaxDeg;
            uint32_t db = 0;
            if (i2 < h->u.e.s1_deg[i1]) {
                uint64_t w2;
                uint32_t b;
                G.edge(h->u.e.s1_node[i1], i2, w2, b);
                const uint64_t q2 = mul_div(h->u.e.s1_q[i1], w2, h->u.e.s1_W[i1]);
                db = G.deg(b);
                seg_insert(h, b, 0, 0, mul_shift32(q2, T));
                if (db == 0) seg_insert(h, b, 1, 2, mul_shift32(q2, cont));
                h->u.e.s2_node[p] = b;
                h->u.e.s2_q[p] = mul_shift32(q2, cont);
                h->u.e.s2_W[p] = db ? G.total(b) : 1ull;
            }
            h->u.e.s2_deg[p] = db;
        }
        __syncwarp();
        // triples packed: pair p owns [pre[p], pre[p + 1])
        uint32_t n3 = 0;  // triples
        for (uint32_t p0 = 0; p0 < np; p0 += 32) {
            uint32_t x = p0 + lane < np ? h->u.e.s2_deg[p0 + lane] : 0u;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
                if (lane >= (uint32_t)o) x += y;
            }
            if (p0 + lane < np) h->u.e.s2_pre[p0 + lane + 1] = n3 + x;
            n3 += __shfl_sync(0xffffffffu, x, 31);
        }
        if (lane == 0) h->u.e.s2_pre[0] = 0;
        __syncwarp();
        for (uint32_t t3 = lane; t3 < n3; t3 += 32) {
            uint32_t lo = 0, hi = np;  // the pair p with pre[p] <= t3 < pre[p + 1]
            while (hi - lo > 1) {
                const uint32_t mid = (lo + hi) >> 1;
                if (h->u.e.s2_pre[mid] <= t3) lo = mid;
                else hi = mid;
            }
            uint64_t w3;
            uint32_t c;
            G.edge(h->u.e.s2_node[lo], t3 - h->u.e.s2_pre[lo], w3, c);
            const uint64_t q3 = mul_div(h->u.e.s2_q[lo], w3, h->u.e.s2_W[lo]);
            seg_insert(h, c, 0, 0, mul_shift32(q3, T));
            seg_insert(h, c, 1, 3, mul_shift32(q3, cont));
        }
        __syncwarp();
        // outcomes of nonzero mass, compacted (the first 64 kept); slots restored
        const uint32_t D = h->count;
        uint32_t K = 0;
        for (uint32_t i0 = 0; i0 < D; i0 += 32) {
            const uint32_t i = i0 + lane;
            unsigned long long k = 0, q = 0;
            if (i < D) {
                const uint32_t s = h->used[i];
                k = h->key[s];
                q = h->val[s];
                h->key[s] = kSegEmpty;
                h->val[s] = 0;
            }
            const bool nzero = i < D && q > 0;
            const uint32_t m = __ballot_sync(0xffffffffu, nzero);
            const uint32_t pos = K + __popc(m & below);
            if (nzero && pos < (uint32_t)kSegMaxOut) {
                h->u.r.sk[pos] = k;
                h->u.r.sq[pos] = q;
            }
            K += __popc(m);
        }
        const bool full = h->full != 0;
        __syncwarp();
        if (lane == 0) {
            h->count = 0;
            h->full = 0;
        }
        if (K == 0 || K > (uint32_t)kSegMaxOut || full) {  // no table: the plain record stays
            __syncwarp();
            continue;
        }
        // canonical order: rank of each key among the K distinct keys (node
        // ids as the caller numbers them)
        unsigned long long mk[2], mq[2], mo[2];
        uint32_t rk[2];
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            const uint32_t i = (uint32_t)e * 32 + lane;
            mk[e] = i < K ? h->u.r.sk[i] : ~0ull;
            mq[e] = i < K ? h->u.r.sq[i] : 0ull;
            mo[e] = i < K ? seg_key_caller(mk[e], order) : mk[e];
            if (i < K) h->u.r.so[i] = mo[e];
        }
        __syncwarp();
        const unsigned long long *cmp = h->u.r.so;
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            uint32_t r = 0;
            for (uint32_t j = 0; j < K; ++j) r += cmp[j] < mo[e];
            rk[e] = r;
        }
        __syncwarp();
#pragma unroll
        for (int e = 0; e < 2; ++e)
            if ((uint32_t)e * 32 + lane < K) {
                h->u.r.sk[rk[e]] = mk[e];
                h->u.r.sq[rk[e]] = mq[e];
            }
        __syncwarp();
        // inclusive prefix of the masses in that order
        unsigned long long cum[2];
        unsigned long long carry = 0;
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            const uint32_t i = (uint32_t)e * 32 + lane;
            unsigned long long x = i < K ? h->u.r.sq[i] : 0ull;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const unsigned long long y = __shfl_up_sync(0xffffffffu, x, o);
                if (lane >= (uint32_t)o) x += y;
            }
            cum[e] = carry + x;
            carry += __shfl_sync(0xffffffffu, x, 31);
        }
        const unsigned long long base = slot[tier ? n - 1 - t : t];
        w_used += K;
        ++w_tables;
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            const uint32_t i = (uint32_t)e * 32 + lane;
            if (i < K) {
                const unsigned long long k = h->u.r.sk[i];
                SegEntry se;
                se.cum = cum[e];
                se.node = code_of_seq(*G.tab, (uint32_t)((k >> 8) & 0x7fffffffull));
                se.mark_len = ((uint32_t)(k >> 63) << 8) | (uint32_t)(k & 0xff);
                ent[base + i] = se;
            }
        }
        // the node's slots (or its single target) now say where its table is
        const uint32_t ent_v = entry_of(*G.tab, v), idx = v - G.tab->e[ent_v].first;
        const TabEntry te = links.tab->e[ent_v];
        if (te.kind == kKindSingle) {
            if (lane == 0) {
                uint32_t *to = reinterpret_cast<uint32_t *>(te.addr) + idx;
                *to = kMarkSeg;
                links.head[to - links.single] = SegHead{pack_word0(base, K), carry};
            }
        } else {
            Sector *at = reinterpret_cast<Sector *>(te.addr) + ((uint64_t)idx << te.kind);
            for (uint32_t b = lane; b < (1u << te.kind); b += 32)
                st_sector(at + b, Sector{{(uint32_t)carry, (uint32_t)(carry >> 32), 0u, 0u, kMarkSeg, (uint32_t)base,
                                          (uint32_t)(base >> 32), K}});
        }
        __syncwarp();
    }
    if (lane == 0 && w_tables) {
        atomicAdd(&ct->used, w_used);
        atomicAdd(&ct->tables, w_tables);
    }
}

template <class E>
static int seg_build_typed(ppr_graph *g, uint32_t T, cudaStream_t st, const RowView<E> &G, uint32_t *list,
                           SegCounters *d_ct)
{
    const int64_t n = g->n;
    const SegLinks links{g->seg.tab, g->seg.single, g->seg.head};
    uint32_t *lbound = nullptr;
    uint64_t *slot = nullptr, *scan_tmp = nullptr;
    auto done = [&](int code) {
        dev_free(lbound, st);
        dev_free(slot, st);
        dev_free(scan_tmp, st);
        return code;
    };
    int rc;
    if ((rc = dev_alloc((void **)&lbound, sizeof(uint32_t) * n, "segment bounds", st)) ||
        (rc = dev_alloc((void **)&slot, sizeof(uint64_t) * (n + 1), "segment slots", st)) ||
        (rc = dev_alloc((void **)&scan_tmp, sizeof(uint64_t) * ((n + kScanTile - 1) / kScanTile + 2), "scan scratch",
                        st)))
        return done(rc);
    cudaError_t e = cudaMemsetAsync(lbound, 0, sizeof(uint32_t) * n, st);  // unlisted positions take no entries
    if (e != cudaSuccess) return done(cuda_fail(e, "memset"));
    const int blocks = (int)std::max<int64_t>(1, std::min<int64_t>((n + 255) / 256, (int64_t)g->ctx->sms * 16));
    k_seg_scan<E><<<blocks, 256, 0, st>>>(G, n, list, lbound, d_ct);
    note_launch();
    exclusive_scan_u32(lbound, n, slot, scan_tmp, st);  // each listed node's slot range in the entry array
    SegCounters hc;
    e = cudaMemcpyAsync(&hc, d_ct, sizeof(hc), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) return done(cuda_fail(e, "segment scan"));
    if ((rc = dev_alloc((void **)&g->seg.entries, sizeof(SegEntry) * (hc.bound > 0 ? hc.bound : 1), "segment tables",
                        st)))
        return done(rc);
    if (hc.listed[0]) {
        constexpr int W = 8;
        const size_t smem = sizeof(SegHash<2 * kSegSmallRaw>) * W;
        e = cudaFuncSetAttribute(k_seg_fill<E, 2 * kSegSmallRaw, W>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)smem);
        if (e != cudaSuccess) return done(cuda_fail(e, "cudaFuncSetAttribute(k_seg_fill)"));
        const int fb = (int)std::min<int64_t>((hc.listed[0] + W - 1) / W, (int64_t)g->ctx->sms * 16);
        k_seg_fill<E, 2 * kSegSmallRaw, W><<<fb, 32 * W, smem, st>>>(G, T, list, 0, n, d_ct, g->seg.entries, links,
                                                                     g->order, slot);
        note_launch();
    }
    if (hc.listed[1]) {
        constexpr int W = 2;
        const size_t smem = sizeof(SegHash<kSegLargeSlots>) * W;
        e = cudaFuncSetAttribute(k_seg_fill<E, kSegLargeSlots, W>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)smem);
        if (e != cudaSuccess) return done(cuda_fail(e, "cudaFuncSetAttribute(k_seg_fill)"));
        const int fb = (int)std::min<int64_t>((hc.listed[1] + W - 1) / W, (int64_t)g->ctx->sms * 8);
        k_seg_fill<E, kSegLargeSlots, W><<<fb, 32 * W, smem, st>>>(G, T, list, 1, n, d_ct, g->seg.entries, links,
                                                                   g->order, slot);
        note_launch();
    }
    e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaMemcpyAsync(&hc, d_ct, sizeof(hc), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) return done(cuda_fail(e, "segment build"));
    g->seg.nodes = (int64_t)hc.tables;
    g->seg.entries_n = (int64_t)hc.used;
    g->seg.entries_cap = (int64_t)hc.bound;
    g->device_bytes += (int64_t)(sizeof(Sector) * g->seg.n_slots + (4 + sizeof(SegHead)) * g->n_single +
                                 sizeof(SegEntry) * hc.bound);
    return done(PPR_OK);
}

static void free_segments(ppr_graph *g, cudaStream_t st)
{
    dev_free(g->seg.tab, st);
    dev_free(g->seg.slots, st);
    dev_free(g->seg.single, st);
    dev_free(g->seg.head, st);
    dev_free(g->seg.entries, st);
    g->seg = SegCache{};
}

int build_segments(ppr_graph *g, uint32_t T, cudaStream_t st)
{
    if (g->seg.T == T && g->seg.tab) return PPR_OK;
    Range range("segment tables");
    free_segments(g, st);
    const int64_t n = g->n;
    uint32_t *list = nullptr;
    SegCounters *d_ct = nullptr;
    int rc;
    auto done = [&](int code) {
        dev_free(list, st);
        dev_free(d_ct, st);
        if (code != PPR_OK) {
            cudaStreamSynchronize(st);
            free_segments(g, st);
        }
        return code;
    };
    // the classes that hold rows of up to eight edges come first among the
    // slots: the segment layout has its own copy of those, and of the single
    // targets, and shares the rest
    const uint32_t small = ranges_log2(kSegMaxDeg, g->lam_bits, g->wide);
    ClassTab tab = g->htab;
    int64_t ns = 0;
    for (uint32_t e = 0; e < kTabEntries; ++e)
        if (tab.e[e].kind <= small) {
            const uint64_t next = e + 1 < kTabEntries && tab.e[e + 1].first != 0xffffffffu ? tab.e[e + 1].first : (uint64_t)n;
            ns = (int64_t)(reinterpret_cast<const Sector *>(tab.e[e].addr) - g->slots) +
                 ((int64_t)(next - tab.e[e].first) << tab.e[e].kind);
        }
    if ((rc = dev_alloc((void **)&list, sizeof(uint32_t) * n, "segment node list", st)) ||
        (rc = dev_alloc((void **)&d_ct, sizeof(SegCounters), "segment counters", st)) ||
        (rc = dev_alloc((void **)&g->seg.tab, sizeof(ClassTab), "segment class table", st)) ||
        (rc = dev_alloc((void **)&g->seg.slots, sizeof(Sector) * std::max<int64_t>(ns, 1), "segment slots", st)) ||
        (rc = dev_alloc((void **)&g->seg.single, sizeof(uint32_t) * std::max<int64_t>(g->n_single, 1), "segment singles",
                        st)) ||
        (rc = dev_alloc((void **)&g->seg.head, sizeof(SegHead) * std::max<int64_t>(g->n_single, 1), "segment heads", st)))
        return done(rc);
    g->seg.n_slots = ns;
    for (TabEntry &t : tab.e) {
        if (t.kind <= small) t.addr += reinterpret_cast<uint64_t>(g->seg.slots) - reinterpret_cast<uint64_t>(g->slots);
        if (t.kind == kKindSingle)
            t.addr += reinterpret_cast<uint64_t>(g->seg.single) - reinterpret_cast<uint64_t>(g->single);
    }
    cudaError_t e = cudaMemsetAsync(d_ct, 0, sizeof(SegCounters), st);
    if (e == cudaSuccess) e = cudaMemcpyAsync(g->seg.tab, &tab, sizeof(tab), cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess && ns > 0)
        e = cudaMemcpyAsync(g->seg.slots, g->slots, sizeof(Sector) * ns, cudaMemcpyDeviceToDevice, st);
    if (e == cudaSuccess && g->n_single > 0)
        e = cudaMemcpyAsync(g->seg.single, g->single, sizeof(uint32_t) * g->n_single, cudaMemcpyDeviceToDevice, st);
    if (e != cudaSuccess) return done(cuda_fail(e, "segment slots"));
    if (g->wide) {
        RowView<WideEdges> G{g->node, WideEdges{(const EdgeW *)g->edges}, g->tab};
        rc = seg_build_typed(g, T, st, G, list, d_ct);
    } else {
        RowView<NarrowEdges> G{g->node, NarrowEdges{(const EdgeN *)g->edges}, g->tab};
        rc = seg_build_typed(g, T, st, G, list, d_ct);
    }
    if (rc != PPR_OK) return done(rc);
    g->seg.T = T;
    return done(PPR_OK);
}

// --------------------------------------------------------- alias tables ----
// Integer Algorithm 1 per row: p_e = d * w_e against a slot capacity of W.
// The pairing order (free in Algorithm 1): y is the first edge of S^l in
// ascending order; x is the edge that has just dropped into S^s if there is
// one, else the next edge of the initial S^s in ascending order.  In that
// order the whole table is a closed form of two running sums -- D_i over the
// small edges of W - p, E_j over the large edges of p - W:
//   small edge i: thr = p, alias = large edge min{j : E_j > D_(i-1)}
//   large edge j (not the last): thr = W - (D_q - E_j) with q = min{q : D_q >= E_j},
//                                alias = large edge j + 1
//   last large edge, edges with p = W: thr = W, alias = itself.
// Rows of at most 32 edges run the pairing rounds serially, one thread per
// row; longer rows compute the closed form: one warp per row with the row in
// shared memory (up to 512 edges), one warp (up to 1,024) or block (up to
// 8,192) per row with scratch in global memory (alias_row_group), and tiles
// of blocks above that.  The limits keep each row's merge to a few dozen
// dependent probes per thread, so no long row is left running alone.

constexpr uint32_t kAliasInline = 32, kAliasSerial = 512, kAliasMid = 1024, kAliasHuge = 8192;
constexpr uint32_t kAliasMaxHuge = 65536;  // rows taken by the tile path; more go to the block tier
constexpr uint32_t kTileEdges = 8192;     // edges per tile block (256 threads x 32)

struct AliasArgs {
    int64_t n;
    const NodeRec *node;  // the narrow layout's records (begin, count, W), by seq
    const EdgeN *edges;
    const uint64_t *off;  // first slot of each row (exclusive scan of degrees)
    AliasNode *anode;     // rows from seq first_node on
    int64_t first_node;
    AliasRec *slots;
    uint2 *ic;            // per slot of a long row: (edge, col) of the small edges from the front,
                          // of the large edges from the back
    uint64_t *sum;        // their running sums D_i / E_j
    uint32_t *list;       // rows per tier: [0, n) one thread, [n, 2n) one warp, [2n, 3n) one block
    uint32_t *counts;     // rows in each list; [3] rows offered to the tile path
    uint2 *huge;          // tile-path rows (node, degree), kAliasMaxHuge entries
};

template <class N>
__device__ __forceinline__ uint32_t row_degree(const N &r) { return (uint32_t)(r.word0 >> 40) & kCountMask; }

// The pairing rounds of one row, serially (row of d >= 2 edges, slots from o).
__device__ void alias_row_serial(const AliasArgs &A, const NodeRec &nr, uint32_t d, uint64_t o)
{
    const uint64_t W = nr.total & 0xffffffffull;
    const uint64_t eb = nr.word0 & kBeginMask;
    auto pw = [&](uint32_t i) -> uint64_t {
        const uint32_t hi = A.edges[eb + i].P, lo = i ? A.edges[eb + i - 1].P : 0u;
        return (uint64_t)d * (hi - lo);
    };
    for (uint32_t i = 0; i < d; ++i) {
        const int32_t c = A.edges[eb + i].col;
        A.slots[o + i] = AliasRec{(uint32_t)W, c, c, (uint32_t)W};
    }
    auto next_small = [&](uint32_t i) { while (i < d && pw(i) >= W) ++i; return i; };
    auto next_large = [&](uint32_t j) { while (j < d && pw(j) <= W) ++j; return j; };
    uint32_t i = next_small(0), j = next_large(0);
    if (j >= d) return;
    uint64_t py = pw(j);  // remaining p of the current large edge
    for (uint32_t guard = 0; guard < 2 * d; ++guard) {
        if (py > W) {  // x = next small edge, y = j
            if (i >= d) break;
            const uint64_t px = pw(i);
            A.slots[o + i].thr = (uint32_t)px;
            A.slots[o + i].alias_col = A.edges[eb + j].col;
            py -= W - px;
            i = next_small(i + 1);
        } else {  // j leaves S^l; if it dropped below W it is the next x
            const uint32_t j2 = next_large(j + 1);
            if (j2 >= d) break;  // py == W here: the last large edge
            if (py < W) {
                A.slots[o + j].thr = (uint32_t)py;
                A.slots[o + j].alias_col = A.edges[eb + j2].col;
            }
            py = pw(j2) - (W - py);
            j = j2;
        }
    }
}

// Node records of the alias layout for every row; rows of at most 32 edges
// are built here, longer ones are listed for their tier.
__global__ void __launch_bounds__(256) k_alias_small(AliasArgs A)
{
    for (int64_t u = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; u < A.n; u += (int64_t)gridDim.x * blockDim.x) {
        const NodeRec nr = A.node[u];
        const uint32_t d = row_degree(nr);
        const uint64_t o = A.off[u];
        if (u >= A.first_node) A.anode[u - A.first_node] = AliasNode{pack_word0(o, d)};
        if (d < 2) continue;
        if (d > kAliasInline) {
            if (d > kAliasHuge) {
                const uint32_t k = atomicAdd(&A.counts[3], 1u);
                if (k < kAliasMaxHuge) {
                    A.huge[k] = make_uint2((uint32_t)u, d);
                    continue;
                }
            }
            const uint32_t tier = d <= kAliasSerial ? 0 : (d <= kAliasMid ? 1 : 2);
            A.list[(int64_t)tier * A.n + atomicAdd(&A.counts[tier], 1u)] = (uint32_t)u;
            continue;
        }
        alias_row_serial(A, nr, d, o);
    }
}

// Rows of 33..512 edges, one warp per row, the row staged in shared memory:
// a coalesced pass classifies the edges, ranks them with ballots and forms
// the running sums D and E with warp scans; each lane then merges a
// contiguous share of the small (and of the large) edges against the other
// sequence, as alias_row_group does, with every probe in shared memory.
constexpr int kSmemWarps = 4;
struct RowSmem {
    int32_t col[kAliasSerial];
    uint16_t idx[kAliasSerial];  // edge of each small (from the front) and large (from the back) entry
    uint64_t sum[kAliasSerial];  // D_i / E_j
};

__global__ void __launch_bounds__(32 * kSmemWarps) k_alias_serial(AliasArgs A)
{
    __shared__ RowSmem sm_all[kSmemWarps];
    RowSmem &sm = sm_all[threadIdx.x >> 5];
    const uint32_t lane = threadIdx.x & 31;
    const uint32_t rows = A.counts[0];
    const uint32_t warps = gridDim.x * kSmemWarps;
    for (uint32_t t = blockIdx.x * kSmemWarps + (threadIdx.x >> 5); t < rows; t += warps) {
        const uint32_t u = A.list[t];
        const NodeRec nr = A.node[u];
        const uint32_t d = row_degree(nr);  // 33..512
        const uint64_t o = A.off[u];
        const uint64_t W = nr.total & 0xffffffffull;
        const uint64_t eb = nr.word0 & kBeginMask;
        uint32_t ns = 0, nl = 0;
        uint64_t Dc = 0, Ec = 0;
        for (uint32_t e0 = 0; e0 < d; e0 += 32) {
            const uint32_t i = e0 + lane;
            uint64_t p = 0;
            int32_t c = 0;
            if (i < d) {
                const EdgeN rec = A.edges[eb + i];
                const uint32_t lo = i ? A.edges[eb + i - 1].P : 0u;
                p = (uint64_t)d * (rec.P - lo);
                c = rec.col;
                sm.col[i] = c;
                A.slots[o + i] = AliasRec{(uint32_t)W, c, c, (uint32_t)W};
            }
            const bool isS = i < d && p < W, isL = i < d && p > W;
            const uint32_t bs = __ballot_sync(0xffffffffu, isS), bl = __ballot_sync(0xffffffffu, isL);
            const uint32_t lt = (1u << lane) - 1;
            uint64_t dv = isS ? W - p : 0ull, ev = isL ? p - W : 0ull;
#pragma unroll
            for (int q = 1; q < 32; q <<= 1) {
                const uint64_t yd = __shfl_up_sync(0xffffffffu, dv, q), ye = __shfl_up_sync(0xffffffffu, ev, q);
                if (lane >= (uint32_t)q) {
                    dv += yd;
                    ev += ye;
                }
            }
            if (isS) {
                const uint32_t k = ns + __popc(bs & lt);
                sm.idx[k] = (uint16_t)i;
                sm.sum[k] = Dc + dv;
            } else if (isL) {
                const uint32_t k = d - 1 - (nl + __popc(bl & lt));
                sm.idx[k] = (uint16_t)i;
                sm.sum[k] = Ec + ev;
            }
            ns += __popc(bs);
            nl += __popc(bl);
            Dc += __shfl_sync(0xffffffffu, dv, 31);
            Ec += __shfl_sync(0xffffffffu, ev, 31);
        }
        __syncwarp();
        const uint32_t a = ns, b = nl;
        if (a > 0 && b > 0 && a + b <= d) {
            auto E = [&](uint32_t j) { return sm.sum[d - 1 - j]; };
            auto D = [&](uint32_t q) { return sm.sum[q]; };
            // small edges t: donor = first large j with E_j > D_(t-1)
            const uint32_t shs = (a + 31) / 32, t0 = min(lane * shs, a), t1 = min(t0 + shs, a);
            if (t0 < t1) {
                uint64_t prev = t0 ? D(t0 - 1) : 0ull;
                uint32_t jl = 0, jh = b - 1;
                while (jl < jh) {
                    const uint32_t mid = (jl + jh) >> 1;
                    if (E(mid) > prev) jh = mid;
                    else jl = mid + 1;
                }
                uint32_t j = jl;
                for (uint32_t tt = t0; tt < t1; ++tt) {
                    while (j + 1 < b && E(j) <= prev) ++j;
                    const uint64_t Dt = D(tt);
                    const uint32_t e = sm.idx[tt];
                    A.slots[o + e].thr = (uint32_t)(W - (Dt - prev));
                    A.slots[o + e].alias_col = sm.col[sm.idx[d - 1 - j]];
                    prev = Dt;
                }
            }
            // large edges j (not the last): q = first small with D_q >= E_j
            const uint32_t nlm = b - 1, shl = (nlm + 31) / 32;
            const uint32_t j0 = min(lane * shl, nlm), j1 = min(j0 + shl, nlm);
            if (j0 < j1) {
                uint64_t Ej = E(j0);
                uint32_t ql = 0, qh = a - 1;
                while (ql < qh) {
                    const uint32_t mid = (ql + qh) >> 1;
                    if (D(mid) >= Ej) qh = mid;
                    else ql = mid + 1;
                }
                uint32_t q = ql;
                for (uint32_t j = j0; j < j1; ++j) {
                    Ej = E(j);
                    while (q + 1 < a && D(q) < Ej) ++q;
                    const uint64_t th = W - (D(q) - Ej);
                    if (th < W) {
                        const uint32_t e = sm.idx[d - 1 - j];
                        A.slots[o + e].thr = (uint32_t)th;
                        A.slots[o + e].alias_col = sm.col[sm.idx[d - 2 - j]];
                    }
                }
            }
        }
        __syncwarp();  // the next row reuses the warp's shared memory
    }
}

// Inclusive scan of three u64 values over a warp (NT = 32) or a block; `tot`
// receives the group totals.  Block form: s holds 3 * (NT / 32) words.
template <int NT>
__device__ __forceinline__ void group_scan3(uint64_t v[3], uint64_t tot[3], uint64_t *s)
{
    const uint32_t lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint64_t y = __shfl_up_sync(0xffffffffu, v[k], o);
            if (lane >= o) v[k] += y;
        }
    }
    if constexpr (NT == 32) {
#pragma unroll
        for (int k = 0; k < 3; ++k) tot[k] = __shfl_sync(0xffffffffu, v[k], 31);
    } else {
        constexpr int NW = NT / 32;
        if (lane == 31)
            for (int k = 0; k < 3; ++k) s[k * NW + wid] = v[k];
        __syncthreads();
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            uint64_t before = 0, all = 0;
            for (int q = 0; q < NW; ++q) {
                const uint64_t t = s[k * NW + q];
                before += q < (int)wid ? t : 0ull;
                all += t;
            }
            v[k] += before;
            tot[k] = all;
        }
        __syncthreads();
    }
}

template <int NT>
__device__ __forceinline__ void group_sync()
{
    if constexpr (NT == 32) __syncwarp();
    else __syncthreads();
}

// Closed-form alias table of one row of d > 32 edges by a group of NT threads
// (rank = thread index within the group).  Each thread owns a contiguous run
// of about d / NT edges: it totals its run, one group scan gives the run's
// starting ranks and sums, and a second walk over the run writes the small
// and large edges with their running sums to scratch.  The partners are then
// a merge of the two sorted sequences D and E: each thread takes a contiguous
// share of the small (and of the large) edges, finds its first partner by
// bisection and advances linearly from there.
template <int NT>
__device__ void alias_row_group(const AliasArgs &A, int64_t u, uint32_t rank, uint64_t *s)
{
    const NodeRec nr = A.node[u];
    const uint32_t d = row_degree(nr);
    const uint64_t o = A.off[u];
    const uint64_t W = nr.total & 0xffffffffull;
    const uint64_t eb = nr.word0 & kBeginMask;
    const uint32_t run = (d + NT - 1) / NT;
    const uint32_t lo = min(rank * run, d), hi = min(lo + run, d);
    // totals of this thread's run
    uint64_t v[3] = {0, 0, 0};  // small | large << 32 counts, sum of W - p, sum of p - W
    {
        uint32_t prevP = lo ? A.edges[eb + lo - 1].P : 0u;
        for (uint32_t i0 = lo; i0 < hi; i0 += 8) {
            uint32_t Pv[8];  // eight loads in flight before their use
#pragma unroll
            for (int q = 0; q < 8; ++q) Pv[q] = i0 + q < hi ? A.edges[eb + i0 + q].P : 0u;
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                if (i0 + q >= hi) break;
                const uint64_t p = (uint64_t)d * (Pv[q] - prevP);
                prevP = Pv[q];
                if (p < W) {
                    v[0] += 1;
                    v[1] += W - p;
                } else if (p > W) {
                    v[0] += 1ull << 32;
                    v[2] += p - W;
                }
            }
        }
    }
    const uint64_t own[3] = {v[0], v[1], v[2]};
    uint64_t tot[3];
    group_scan3<NT>(v, tot, s);
    uint64_t ks = (v[0] - own[0]) & 0xffffffffull, kl = (v[0] - own[0]) >> 32;
    uint64_t Dr = v[1] - own[1], Er = v[2] - own[2];
    {
        uint32_t prevP = lo ? A.edges[eb + lo - 1].P : 0u;
        for (uint32_t i0 = lo; i0 < hi; i0 += 8) {
            EdgeN rv[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                if (i0 + q < hi) rv[q] = A.edges[eb + i0 + q];
                else rv[q] = EdgeN{0u, 0};
            }
#pragma unroll
            for (int q = 0; q < 8; ++q) {
                const uint32_t i = i0 + q;
                if (i >= hi) break;
                const EdgeN rec = rv[q];
                const uint64_t p = (uint64_t)d * (rec.P - prevP);
                prevP = rec.P;
                A.slots[o + i] = AliasRec{(uint32_t)W, rec.col, rec.col, (uint32_t)W};
                if (p < W && ks < d) {
                    Dr += W - p;
                    A.ic[o + ks] = make_uint2(i, (uint32_t)rec.col);
                    A.sum[o + ks] = Dr;
                    ++ks;
                } else if (p > W && kl < d) {
                    Er += p - W;
                    A.ic[o + d - 1 - kl] = make_uint2(i, (uint32_t)rec.col);
                    A.sum[o + d - 1 - kl] = Er;
                    ++kl;
                }
            }
        }
    }
    group_sync<NT>();
    const uint32_t a = (uint32_t)(tot[0] & 0xffffffffull), b = (uint32_t)(tot[0] >> 32);
    if (a == 0 || b == 0 || (uint64_t)a + b > d) return;  // every p equals W (the sums force a > 0 iff b > 0)
    auto E = [&](uint32_t j) { return A.sum[o + d - 1 - j]; };
    auto D = [&](uint32_t q) { return A.sum[o + q]; };
    auto large_col = [&](uint32_t j) { return (int32_t)A.ic[o + d - 1 - j].y; };
    // small edges t in [t0, t1): donor = first large j with E_j > D_(t-1)
    {
        const uint32_t share = (a + NT - 1) / NT;
        const uint32_t t0 = min(rank * share, a), t1 = min(t0 + share, a);
        if (t0 < t1) {
            uint64_t prev = t0 ? D(t0 - 1) : 0ull;
            uint32_t jl = 0, jh = b - 1;
            while (jl < jh) {
                const uint32_t mid = (jl + jh) >> 1;
                if (E(mid) > prev) jh = mid;
                else jl = mid + 1;
            }
            uint32_t j = jl;
            for (uint32_t t = t0; t < t1; ++t) {
                while (j + 1 < b && E(j) <= prev) ++j;
                const uint64_t Dt = D(t);
                const uint32_t e = A.ic[o + t].x;
                A.slots[o + e].thr = (uint32_t)(W - (Dt - prev));
                A.slots[o + e].alias_col = large_col(j);
                prev = Dt;
            }
        }
    }
    // large edges j in [j0, j1) (not the last): q = first small with D_q >= E_j
    {
        const uint32_t nl = b - 1, share = (nl + NT - 1) / NT;
        const uint32_t j0 = min(rank * share, nl), j1 = min(j0 + share, nl);
        if (j0 < j1) {
            uint64_t Ej = E(j0);
            uint32_t ql = 0, qh = a - 1;
            while (ql < qh) {
                const uint32_t mid = (ql + qh) >> 1;
                if (D(mid) >= Ej) qh = mid;
                else ql = mid + 1;
            }
            uint32_t q = ql;
            for (uint32_t j = j0; j < j1; ++j) {
                Ej = E(j);
                while (q + 1 < a && D(q) < Ej) ++q;
                const uint64_t th = W - (D(q) - Ej);
                if (th < W) {
                    const uint32_t e = A.ic[o + d - 1 - j].x;
                    A.slots[o + e].thr = (uint32_t)th;
                    A.slots[o + e].alias_col = large_col(j + 1);
                }
            }
        }
    }
}

__global__ void __launch_bounds__(256) k_alias_mid(AliasArgs A)
{
    const uint32_t lane = threadIdx.x & 31;
    const int64_t warps = (int64_t)gridDim.x * (blockDim.x >> 5);
    const uint32_t rows = A.counts[1];
    for (int64_t t = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; t < rows; t += warps)
        alias_row_group<32>(A, A.list[A.n + t], lane, nullptr);
}

__global__ void __launch_bounds__(512) k_alias_big(AliasArgs A)
{
    __shared__ uint64_t s[3 * 16];
    const uint32_t rows = A.counts[2];
    for (uint32_t t = blockIdx.x; t < rows; t += gridDim.x) {
        alias_row_group<512>(A, A.list[2 * A.n + t], threadIdx.x, s);
        __syncthreads();
    }
}

// ------------------------------------------------ alias tables: tile path ----
// Rows above kAliasHuge edges are cut into tiles of kTileEdges edges, one
// block per tile, so a hub does not leave one block working while the GPU
// idles: (1) every tile totals its small/large counts and running-sum parts,
// (2) one warp per row scans its tiles' totals, (3) every tile writes its
// small and large edges with their running sums to scratch, (4) merge chunks
// of kTileEdges small (or large) edges each find their partners as in
// alias_row_group.

struct HugeRow {
    uint32_t u, d;
    uint32_t tile0, ntiles;  // tiles of the row in the tile table
    uint32_t chunk0;         // first merge chunk (2 * ntiles chunks: small edges, then large edges)
};

struct TileVal {
    uint64_t cnt, D, E;  // small | large << 32 counts, sum of W - p, sum of p - W
};

struct TileArgs {
    AliasArgs A;
    const HugeRow *rows;
    uint32_t nrows;
    const uint2 *tiles;      // (row index, first edge of the tile within the row)
    TileVal *tile_val;       // per tile: its totals, then (after the row scan) its exclusive offsets
    ulonglong2 *row_ab;      // per row: small count, large count
};

// Per-thread run of up to 32 edges of a tile: fills the three totals.
__device__ __forceinline__ void tile_run_totals(const AliasArgs &A, uint64_t eb, uint32_t d, uint64_t W, uint32_t lo,
                                                uint32_t hi, uint64_t v[3])
{
    uint32_t prevP = lo ? A.edges[eb + lo - 1].P : 0u;
    for (uint32_t i0 = lo; i0 < hi; i0 += 8) {
        uint32_t Pv[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) Pv[q] = i0 + q < hi ? A.edges[eb + i0 + q].P : 0u;
#pragma unroll
        for (int q = 0; q < 8; ++q) {
            if (i0 + q >= hi) break;
            const uint64_t p = (uint64_t)d * (Pv[q] - prevP);
            prevP = Pv[q];
            if (p < W) {
                v[0] += 1;
                v[1] += W - p;
            } else if (p > W) {
                v[0] += 1ull << 32;
                v[2] += p - W;
            }
        }
    }
}

__global__ void __launch_bounds__(256) k_alias_tile_totals(TileArgs T)
{
    __shared__ uint64_t s[3 * 8];
    const AliasArgs &A = T.A;
    const uint2 tl = T.tiles[blockIdx.x];
    const HugeRow hr = T.rows[tl.x];
    const NodeRec nr = A.node[hr.u];
    const uint64_t W = nr.total & 0xffffffffull;
    const uint64_t eb = nr.word0 & kBeginMask;
    const uint32_t end = min(tl.y + kTileEdges, hr.d);
    const uint32_t lo = min(tl.y + threadIdx.x * 32, end), hi = min(lo + 32, end);
    uint64_t v[3] = {0, 0, 0};
    tile_run_totals(A, eb, hr.d, W, lo, hi, v);
    uint64_t tot[3];
    group_scan3<256>(v, tot, s);
    if (threadIdx.x == 0) T.tile_val[blockIdx.x] = TileVal{tot[0], tot[1], tot[2]};
}

// One warp per row: exclusive scan of its tiles' totals (in place), row counts.
__global__ void k_alias_tile_scan(TileArgs T)
{
    const uint32_t r = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    if (r >= T.nrows) return;
    const uint32_t lane = threadIdx.x & 31;
    const HugeRow hr = T.rows[r];
    uint64_t carry[3] = {0, 0, 0};
    for (uint32_t t0 = 0; t0 < hr.ntiles; t0 += 32) {
        const uint32_t t = t0 + lane;
        TileVal tv{0, 0, 0};
        if (t < hr.ntiles) tv = T.tile_val[hr.tile0 + t];
        uint64_t v[3] = {tv.cnt, tv.D, tv.E}, tot[3];
        const uint64_t own[3] = {v[0], v[1], v[2]};
        group_scan3<32>(v, tot, nullptr);
        if (t < hr.ntiles)
            T.tile_val[hr.tile0 + t] = TileVal{carry[0] + v[0] - own[0], carry[1] + v[1] - own[1],
                                               carry[2] + v[2] - own[2]};
        for (int k = 0; k < 3; ++k) carry[k] += tot[k];
    }
    if (lane == 0) T.row_ab[r] = make_ulonglong2(carry[0] & 0xffffffffull, carry[0] >> 32);
}

__global__ void __launch_bounds__(256) k_alias_tile_write(TileArgs T)
{
    __shared__ uint64_t s[3 * 8];
    const AliasArgs &A = T.A;
    const uint2 tl = T.tiles[blockIdx.x];
    const HugeRow hr = T.rows[tl.x];
    const uint32_t d = hr.d;
    const NodeRec nr = A.node[hr.u];
    const uint64_t W = nr.total & 0xffffffffull;
    const uint64_t eb = nr.word0 & kBeginMask;
    const uint64_t o = A.off[hr.u];
    const uint32_t end = min(tl.y + kTileEdges, d);
    const uint32_t lo = min(tl.y + threadIdx.x * 32, end), hi = min(lo + 32, end);
    uint64_t v[3] = {0, 0, 0};
    tile_run_totals(A, eb, d, W, lo, hi, v);
    const uint64_t own[3] = {v[0], v[1], v[2]};
    uint64_t tot[3];
    group_scan3<256>(v, tot, s);
    const TileVal base = T.tile_val[blockIdx.x];  // the tile's exclusive offsets within the row
    uint64_t ks = (base.cnt & 0xffffffffull) + ((v[0] - own[0]) & 0xffffffffull);
    uint64_t kl = (base.cnt >> 32) + ((v[0] - own[0]) >> 32);
    uint64_t Dr = base.D + v[1] - own[1], Er = base.E + v[2] - own[2];
    uint32_t prevP = lo ? A.edges[eb + lo - 1].P : 0u;
    for (uint32_t i = lo; i < hi; ++i) {
        const EdgeN rec = A.edges[eb + i];
        const uint64_t p = (uint64_t)d * (rec.P - prevP);
        prevP = rec.P;
        A.slots[o + i] = AliasRec{(uint32_t)W, rec.col, rec.col, (uint32_t)W};
        if (p < W && ks < d) {
            Dr += W - p;
            A.ic[o + ks] = make_uint2(i, (uint32_t)rec.col);
            A.sum[o + ks] = Dr;
            ++ks;
        } else if (p > W && kl < d) {
            Er += p - W;
            A.ic[o + d - 1 - kl] = make_uint2(i, (uint32_t)rec.col);
            A.sum[o + d - 1 - kl] = Er;
            ++kl;
        }
    }
}

// Merge chunk c of a row: chunks [0, ntiles) cover small edges
// [c * kTileEdges, ...), chunks [ntiles, 2 ntiles) cover large edges (the
// last large edge keeps thr = W).  Each thread takes 32 consecutive ones.
__global__ void __launch_bounds__(256) k_alias_tile_merge(TileArgs T)
{
    const AliasArgs &A = T.A;
    uint32_t lo = 0, hi = T.nrows;  // row of this chunk: last row with chunk0 <= blockIdx.x
    while (hi - lo > 1) {
        const uint32_t mid = (lo + hi) >> 1;
        if (T.rows[mid].chunk0 <= blockIdx.x) lo = mid;
        else hi = mid;
    }
    const HugeRow hr = T.rows[lo];
    const uint32_t c = blockIdx.x - hr.chunk0;
    if (c >= 2 * hr.ntiles) return;
    const ulonglong2 ab = T.row_ab[lo];
    const uint32_t a = (uint32_t)ab.x, b = (uint32_t)ab.y, d = hr.d;
    if (a == 0 || b == 0 || (uint64_t)a + b > d) return;
    const NodeRec nr = A.node[hr.u];
    const uint64_t W = nr.total & 0xffffffffull;
    const uint64_t o = A.off[hr.u];
    auto E = [&](uint32_t j) { return A.sum[o + d - 1 - j]; };
    auto D = [&](uint32_t q) { return A.sum[o + q]; };
    if (c < hr.ntiles) {  // small edges t in [t0, t1): donor = first large j with E_j > D_(t-1)
        const uint32_t t0 = min(c * kTileEdges + threadIdx.x * 32, a), t1 = min(t0 + 32, min((c + 1) * kTileEdges, a));
        if (t0 >= t1) return;
        uint64_t prev = t0 ? D(t0 - 1) : 0ull;
        uint32_t jl = 0, jh = b - 1;
        while (jl < jh) {
            const uint32_t mid = (jl + jh) >> 1;
            if (E(mid) > prev) jh = mid;
            else jl = mid + 1;
        }
        uint32_t j = jl;
        for (uint32_t t = t0; t < t1; ++t) {
            while (j + 1 < b && E(j) <= prev) ++j;
            const uint64_t Dt = D(t);
            const uint32_t e = A.ic[o + t].x;
            A.slots[o + e].thr = (uint32_t)(W - (Dt - prev));
            A.slots[o + e].alias_col = (int32_t)A.ic[o + d - 1 - j].y;
            prev = Dt;
        }
    } else {  // large edges j in [j0, j1), not the last: q = first small with D_q >= E_j
        const uint32_t cl = c - hr.ntiles, nl = b - 1;
        const uint32_t j0 = min(cl * kTileEdges + threadIdx.x * 32, nl), j1 = min(j0 + 32, min((cl + 1) * kTileEdges, nl));
        if (j0 >= j1) return;
        uint64_t Ej = E(j0);
        uint32_t ql = 0, qh = a - 1;
        while (ql < qh) {
            const uint32_t mid = (ql + qh) >> 1;
            if (D(mid) >= Ej) qh = mid;
            else ql = mid + 1;
        }
        uint32_t q = ql;
        for (uint32_t j = j0; j < j1; ++j) {
            Ej = E(j);
            while (q + 1 < a && D(q) < Ej) ++q;
            const uint64_t th = W - (D(q) - Ej);
            if (th < W) {
                const uint32_t e = A.ic[o + d - 1 - j].x;
                A.slots[o + e].thr = (uint32_t)th;
                A.slots[o + e].alias_col = (int32_t)A.ic[o + d - 2 - j].y;
            }
        }
    }
}

__global__ void k_alias_degrees(int64_t n, const NodeRec *node, uint32_t *deg)
{
    for (int64_t u = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; u < n; u += (int64_t)gridDim.x * blockDim.x)
    {
        const uint32_t d = row_degree(node[u]);
        deg[u] = d >= 2 ? d : 0;  // walks find a single edge's target in the layout's own array
    }
}

int build_alias(ppr_graph *g, cudaStream_t st)
{
    if (g->alias.tab) return PPR_OK;
    Range range("alias tables");
    if (g->wide) {
        set_error("the alias sampler needs every row total below 2^32");
        return PPR_ENOTSUP;
    }
    const int64_t n = g->n, m = std::max<int64_t>(g->m, 1);
    const int64_t tiles = (n + kScanTile - 1) / kScanTile;
    uint32_t *deg = nullptr, *list = nullptr, *counts = nullptr;
    uint2 *ic = nullptr, *huge = nullptr, *d_tiles = nullptr;
    uint64_t *off = nullptr, *tmp = nullptr, *sum = nullptr;
    HugeRow *d_rows = nullptr;
    TileVal *tile_val = nullptr;
    ulonglong2 *row_ab = nullptr;
    int rc;
    auto cleanup = [&]() {
        dev_free(deg, st);
        dev_free(off, st);
        dev_free(tmp, st);
        dev_free(ic, st);
        dev_free(sum, st);
        dev_free(list, st);
        dev_free(counts, st);
        dev_free(huge, st);
        dev_free(d_rows, st);
        dev_free(d_tiles, st);
        dev_free(tile_val, st);
        dev_free(row_ab, st);
    };
    auto fail = [&](int code) {
        cudaStreamSynchronize(st);
        cleanup();
        dev_free(g->alias.tab, st);
        dev_free(g->alias.node, st);
        dev_free(g->alias.slots, st);
        g->alias = AliasCache{};
        return code;
    };
    if ((rc = dev_alloc((void **)&deg, sizeof(uint32_t) * n, "alias degrees", st)) ||
        (rc = dev_alloc((void **)&off, sizeof(uint64_t) * (n + 1), "alias offsets", st)) ||
        (rc = dev_alloc((void **)&tmp, sizeof(uint64_t) * (tiles + 2), "scan scratch", st)) ||
        (rc = dev_alloc((void **)&ic, sizeof(uint2) * m, "alias scratch", st)) ||
        (rc = dev_alloc((void **)&sum, sizeof(uint64_t) * m, "alias scratch", st)) ||
        (rc = dev_alloc((void **)&list, sizeof(uint32_t) * 3 * n, "long-row lists", st)) ||
        (rc = dev_alloc((void **)&counts, sizeof(uint32_t) * 4, "long-row counts", st)) ||
        (rc = dev_alloc((void **)&huge, sizeof(uint2) * kAliasMaxHuge, "tile-path rows", st)))
        return cleanup(), rc;
    // the rows classed by degree have theirs one after the other, in seq order;
    // the others, which follow, are looked up in node records
    ClassTab tab = g->htab;
    int64_t first_node = n, slot = 0;
    for (uint32_t e = 0; e < kTabEntries && tab.e[e].first != 0xffffffffu; ++e)
        if (tab.e[e].kind < kKindSingle && g->degree[e] == 0) {
            first_node = tab.e[e].first;
            break;
        }
    if ((rc = dev_alloc((void **)&g->alias.node, sizeof(AliasNode) * std::max<int64_t>(n - first_node, 1),
                        "alias node records", st)) ||
        (rc = dev_alloc((void **)&g->alias.slots, sizeof(AliasRec) * m, "alias slots", st)))
        return fail(rc);
    for (uint32_t e = 0; e < kTabEntries && tab.e[e].first != 0xffffffffu; ++e) {
        TabEntry &t = tab.e[e];
        if (t.kind >= kKindSingle) continue;
        if (g->degree[e]) {
            const int64_t next = e + 1 < kTabEntries && tab.e[e + 1].first != 0xffffffffu ? (int64_t)tab.e[e + 1].first : n;
            t.kind = g->degree[e];
            t.addr = reinterpret_cast<uint64_t>(g->alias.slots + slot);
            slot += (next - (int64_t)t.first) * g->degree[e];
        } else {
            t.kind = kKindLookup;
            t.addr = reinterpret_cast<uint64_t>(g->alias.node + ((int64_t)t.first - first_node));
        }
    }
    cudaError_t e = cudaMemsetAsync(counts, 0, sizeof(uint32_t) * 4, st);
    if (e != cudaSuccess) return fail(cuda_fail(e, "memset"));
    const int blocks = (int)std::max<int64_t>(1, std::min<int64_t>((n + 255) / 256, (int64_t)g->ctx->sms * 16));
    k_alias_degrees<<<blocks, 256, 0, st>>>(n, g->node, deg);
    note_launch();
    exclusive_scan_u32(deg, n, off, tmp, st);
    AliasArgs A{n, g->node, (const EdgeN *)g->edges, off, g->alias.node, first_node, g->alias.slots, ic,
                sum, list, counts, huge};
    k_alias_small<<<blocks, 256, 0, st>>>(A);
    note_launch();
    // rows for the tile path: their count and degrees decide the tile grid
    uint32_t hc[4] = {0, 0, 0, 0};
    e = cudaMemcpyAsync(hc, counts, sizeof(hc), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) return fail(cuda_fail(e, "alias build"));
    const uint32_t nh = std::min(hc[3], kAliasMaxHuge);
    if (nh > 0) {
        std::vector<uint2> hl(nh);
        e = cudaMemcpy(hl.data(), huge, sizeof(uint2) * nh, cudaMemcpyDeviceToHost);
        if (e != cudaSuccess) return fail(cuda_fail(e, "alias build"));
        std::vector<HugeRow> rows(nh);
        std::vector<uint2> tl;
        uint32_t chunks = 0;
        for (uint32_t r = 0; r < nh; ++r) {
            const uint32_t d = hl[r].y, nt = (d + kTileEdges - 1) / kTileEdges;
            rows[r] = HugeRow{hl[r].x, d, (uint32_t)tl.size(), nt, chunks};
            for (uint32_t t = 0; t < nt; ++t) tl.push_back(make_uint2(r, t * kTileEdges));
            chunks += 2 * nt;
        }
        const uint32_t nt = (uint32_t)tl.size();
        if ((rc = dev_alloc((void **)&d_rows, sizeof(HugeRow) * nh, "tile-path rows", st)) ||
            (rc = dev_alloc((void **)&d_tiles, sizeof(uint2) * nt, "tile table", st)) ||
            (rc = dev_alloc((void **)&tile_val, sizeof(TileVal) * nt, "tile totals", st)) ||
            (rc = dev_alloc((void **)&row_ab, sizeof(ulonglong2) * nh, "tile-path counts", st)))
            return fail(rc);
        e = cudaMemcpyAsync(d_rows, rows.data(), sizeof(HugeRow) * nh, cudaMemcpyHostToDevice, st);
        if (e == cudaSuccess) e = cudaMemcpyAsync(d_tiles, tl.data(), sizeof(uint2) * nt, cudaMemcpyHostToDevice, st);
        if (e != cudaSuccess) return fail(cuda_fail(e, "tile table upload"));
        TileArgs T{A, d_rows, nh, d_tiles, tile_val, row_ab};
        k_alias_tile_totals<<<nt, 256, 0, st>>>(T);
        note_launch();
        k_alias_tile_scan<<<(nh + 7) / 8, 256, 0, st>>>(T);
        note_launch();
        k_alias_tile_write<<<nt, 256, 0, st>>>(T);
        note_launch();
        k_alias_tile_merge<<<chunks, 256, 0, st>>>(T);
        note_launch();
        // the host vectors must outlive the asynchronous uploads
        e = cudaStreamSynchronize(st);
        if (e != cudaSuccess) return fail(cuda_fail(e, "alias build"));
    }
    if (hc[0]) {
        k_alias_serial<<<g->ctx->sms * 16, 32 * kSmemWarps, 0, st>>>(A);
        note_launch();
    }
    if (hc[1]) {
        k_alias_mid<<<g->ctx->sms * 8, 256, 0, st>>>(A);
        note_launch();
    }
    if (hc[2]) {
        k_alias_big<<<(int)std::min<uint32_t>(hc[2], (uint32_t)g->ctx->sms * 2), 512, 0, st>>>(A);
        note_launch();
    }
    e = cudaGetLastError();
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (e != cudaSuccess) return fail(cuda_fail(e, "alias build"));
    ClassTab *d_tab = nullptr;
    if ((rc = dev_alloc((void **)&d_tab, sizeof(ClassTab), "alias class table", st))) return fail(rc);
    e = cudaMemcpyAsync(d_tab, &tab, sizeof(tab), cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    g->alias.tab = d_tab;
    g->alias.nodes = n - first_node;
    if (e != cudaSuccess) return fail(cuda_fail(e, "alias class table"));
    cleanup();
    g->device_bytes += (int64_t)(sizeof(AliasNode) * (n - first_node) + sizeof(AliasRec) * m);
    return PPR_OK;
}

}  // namespace ppr
