// walk.cu -- the batch walker kernels (one step of a walk: walk_step.cuh).
//
// k_walk_plain:      one thread per walk, endpoint to HBM (baseline).
// k_walk_persistent: persistent warps pull chunks of walks from a global
//                    queue and refill lanes as walks end (the paper's
//                    pipelines keep the cluster busy the same way).
// Both write one endpoint per walk to HBM; k_aggregate (aggregate.cuh) then
// turns each source's R endpoints into its count row and top-k.
#include <algorithm>
#include <atomic>
#include <mutex>

#include "ppr_host.h"
#include "scan.cuh"
#include "aggregate.cuh"
#include "walk_step.cuh"

namespace ppr {

__device__ __forceinline__ void warp_add(unsigned long long *dst, uint32_t v)
{
    unsigned long long s = v;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0 && s) atomicAdd(dst, s);
}

template <bool STATS>
__device__ __forceinline__ void warp_add_tally(unsigned long long *dst, const Tally &t)
{
    warp_add(dst, t.steps);
    if (STATS) {
        warp_add(dst + 2, t.sectors);
        warp_add(dst + 5, t.model);
    }
}

// Resident 256-thread blocks per SM asked of ptxas.  Narrow: 6 (38 registers;
// 8 blocks at 32: 256-graph batch 18.75 against 18.55 ms, R-MAT scale-24 job
// 103.7 against 102.9).  Wide: 8 (scale 18 with amounts as weights, 2.20 -> 2.08
// ms).  Alias: 8 (scale 20 5.37 against 5.47 ms; a quarter of scale 24 level).
template <class E>
constexpr int kWalkBlocks = E::kWide || E::kAlias ? 8 : 6;

// ------------------------------------------------------------ plain (K4) ----
template <class E, bool SEG, bool STATS>
__global__ void __launch_bounds__(256, kWalkBlocks<E>) k_walk_plain(KParams p)
{
    __shared__ ClassTab tab;
    load_tab(tab, p.tab);
    const uint64_t S = (uint64_t)(p.s_end - p.s_begin);
    const uint64_t total = S * p.R;
    Tally tl;
    for (uint64_t t = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; t < total;
         t += (uint64_t)gridDim.x * blockDim.x) {
        const uint64_t i = t / p.R;
        const uint32_t j = (uint32_t)(t - i * p.R);
        const uint32_t src = p.src_list ? p.src_list[i] : (uint32_t)(p.s_begin + (int64_t)i);
        uint32_t ctr_base = 0, tag = p.tag;
        if (p.inst_off) {  // batched graph: the source's instance gives counter base and tag
            int32_t lo = 0, hi = p.instances;
            while (hi - lo > 1) {
                const int32_t mid = (lo + hi) >> 1;
                if (p.inst_off[mid] <= (int64_t)src) lo = mid;
                else hi = mid;
            }
            ctr_base = (uint32_t)p.inst_off[lo];
            tag = (uint32_t)lo;
        }
        // the draw is keyed by the caller's source id; the walk starts (and
        // restarts) at its node of the layout
        const uint32_t s0 = p.code_of[src];
        uint32_t k = 0, u = s0;
        Pending pend;
        while (!walk_step<E, SEG, STATS>(p, tab, p.key, p.T, s0, src - ctr_base, j, tag, k, u, pend, tl)) {
        }
        if (!SEG) tl.steps += k;
        p.ends[t] = u;
    }
    warp_add_tally<STATS>(p.steps, tl);
}

// ------------------------------------------------------- persistent (K5) ----
// Persistent warps.  Each warp pulls chunks of walks from a global queue (one
// atomic per chunk) and keeps all 32 lanes busy: a lane whose walk ends takes
// the next walk of the warp's chunk at once, so a warp never waits for the
// longest of 32 geometric walk lengths (the paper's pipelines keep the cluster
// busy the same way: new walks start while old ones finish).  Walks start in
// order, so those of one source start close together and share the loads of
// its row (with walks dealt out to lanes in advance, l, l + 32, ..., lanes
// drift apart and the scale-24 walker took 120 ms, not 93).  Steps run in
// lockstep, one load each (walk_step).  Endpoints go to the per-walk buffer as
// node codes, reduced per source by k_aggregate.
struct WarpChunk {
    uint32_t base, ctr_base, tag;  // first position, counter base, tag
    uint32_t j0;                   // walk index (within source `base`) of the chunk's first walk
    uint2 src[32];                 // counter id and code of the chunk's sources
};
// A chunk's sources are read when a warp takes it, one a lane, so that no
// refill waits for them (256-graph batch 18.91 -> 18.55 ms, R-MAT scale-24 job
// 103.8 -> 102.9, scale 20 8.10 -> 8.01; the wide walker, short of registers,
// reads them as it starts walks: 2.200 ms, staged 2.227).  So a chunk has at
// most 31 whole sources, or parts of 32, also where that is far less than 400
// walks (R up to 12): with places for 63 or 127 sources scale 20 takes 568 or
// 599 us, not 558, at R 2, 1,009 or 1,011, not 957, at R 6, and its alias
// walker, which loses L1 to the places, 8.08 or 8.20 ms, not 7.52, at R 100.
constexpr uint32_t kChunkSources = 31;

__device__ __forceinline__ uint32_t div_by_R(uint32_t w, uint64_t magic)
{
    return (uint32_t)(((uint64_t)w * magic) >> 40);  // exact for w < 2^20, R <= 4096
}

template <class E, bool SEG, bool STATS>
__global__ void __launch_bounds__(256, kWalkBlocks<E>) k_walk_persistent(KParams p)
{
    __shared__ WarpChunk chunk_all[8];
    __shared__ ClassTab tab;
    __shared__ unsigned long long nchunks;
    if (threadIdx.x == 0) nchunks = p.nchunks_dev ? *p.nchunks_dev : p.nchunks;
    load_tab(tab, p.tab);
    const uint32_t lane = threadIdx.x & 31;
    WarpChunk &wc = chunk_all[threadIdx.x >> 5];
    uint32_t issued = 0, total = 0;  // uniform: walks of the chunk handed out, and its walks
    bool queue_empty = false;        // uniform
    bool active = false;
    uint32_t src = 0, sctr = 0, j = 0, k = 0, u = 0, tag = 0, pos = 0;
    Pending pend;
    Tally tl;

    for (;;) {
        uint32_t idle = __ballot_sync(0xffffffffu, !active);
        // refill once p.refill lanes are idle, then every idle lane
        if ((uint32_t)__popc(idle) >= p.refill) {
            while (idle) {
                if (issued == total) {
                    if (queue_empty) break;
                    unsigned long long c = 0;
                    if (lane == 0) c = atomicAdd(p.queue, 1ull);
                    c = __shfl_sync(0xffffffffu, c, 0);
                    if (c >= nchunks) {
                        queue_empty = true;
                        break;
                    }
                    uint32_t base, ctr_base = 0, ctag = p.tag, j0 = 0, nsrc;
                    if (p.chunks) {  // whole sources of one instance
                        const int4 d = p.chunks[c];
                        base = (uint32_t)d.x;
                        ctr_base = (uint32_t)d.w;
                        ctag = (uint32_t)d.z;
                        nsrc = (uint32_t)d.y;
                        total = nsrc * p.R;
                    } else {  // walks [c * CW, ...) of the whole launch
                        const uint64_t b = c * (uint64_t)p.CW, i0 = b / p.R;
                        base = (uint32_t)i0;
                        j0 = (uint32_t)(b - i0 * p.R);
                        total = (uint32_t)min((uint64_t)p.CW, p.walks - b);
                        nsrc = div_by_R(j0 + total - 1, p.r_magic) + 1;
                    }
                    __syncwarp();  // the walks of the chunk before have been started
                    if (lane == 0) {
                        wc.base = base;
                        wc.ctr_base = ctr_base;
                        wc.tag = ctag;
                        wc.j0 = j0;
                    }
                    if (!E::kWide && lane < nsrc) {  // draws are keyed by the caller's source id; walks start at its node of the layout
                        const uint32_t id = p.src_list ? p.src_list[base + lane] : (uint32_t)(p.s_begin + base + lane);
                        wc.src[lane] = make_uint2(id - ctr_base, p.code_of[id]);
                    }
                    issued = 0;
                    __syncwarp();
                }
                const uint32_t n = issued + __popc(idle & ((1u << lane) - 1));  // the walk this lane would take
                if (!active && n < total) {
                    const uint32_t w = wc.j0 + n;  // < 2^20: a chunk <= 2^19 walks, j0 < R <= 4096
                    const uint32_t i = div_by_R(w, p.r_magic);
                    j = w - i * p.R;
                    pos = wc.base + i;
                    if constexpr (!E::kWide) {
                        const uint2 s = wc.src[i];
                        sctr = s.x;
                        src = s.y;
                    } else {
                        src = p.src_list ? p.src_list[pos] : (uint32_t)(p.s_begin + pos);
                        sctr = src - wc.ctr_base;
                        src = p.code_of[src];
                    }
                    tag = wc.tag;
                    k = 0;
                    u = src;
                    active = true;
                }
                const uint32_t want = __popc(idle);
                if (want <= total - issued) {
                    issued += want;
                    break;
                }
                issued = total;  // the lanes left take walks of the next chunk
                __syncwarp();
                idle = __ballot_sync(0xffffffffu, !active);
            }
            if (queue_empty && __ballot_sync(0xffffffffu, active) == 0) break;  // queue drained, every walk done
        }
        if (active && walk_step<E, SEG, STATS>(p, tab, p.key, p.T, src, sctr, j, tag, k, u, pend, tl)) {
            const uint64_t slot = (uint64_t)pos * p.R + j;
#ifdef PPR_CHECKED
            if (slot >= (uint64_t)(p.s_end - p.s_begin) * p.R) atomicOr(p.err, 8ull);
            else
#endif
            p.ends[slot] = u;
            if (!SEG) tl.steps += k;
            active = false;
        }
    }
    warp_add_tally<STATS>(p.steps, tl);
}

// ------------------------------------------------------------- launcher ----

// Events around a walker launch, for the walker-only device time.
static int walker_event(ppr_result *r, cudaStream_t st)
{
    if (!r) return PPR_OK;  // allocation-free runs record no events
    cudaEvent_t ev;
    PPR_CUDA(cudaEventCreate(&ev));
    r->walk_events.push_back(ev);
    PPR_CUDA(cudaEventRecord(ev, st));
    return PPR_OK;
}

template <class E, bool SEG, bool STATS>
static int launch_typed(ppr_ctx *ctx, const KParams &kp, const RunPlan &plan, int64_t S, cudaStream_t st,
                        ppr_result *r)
{
    int rc;
    if (plan.kernel == PPR_KERNEL_PLAIN) {
        uint64_t total = (uint64_t)S * kp.R;
        int blocks = (int)std::min<uint64_t>((total + 255) / 256, (uint64_t)ctx->sms * 64);
        if (blocks < 1) blocks = 1;
        if ((rc = walker_event(r, st))) return rc;
        k_walk_plain<E, SEG, STATS><<<blocks, 256, 0, st>>>(kp);
        note_launch();
        PPR_CUDA(cudaGetLastError());
        if ((rc = walker_event(r, st))) return rc;
        return launch_aggregate(ctx, AggParams{kp.ends, kp.R, kp.P2, S, kp.out_row0, kp.out, kp.order, kp.tab}, st);
    }
    // walkers per CTA: 32 * warps_per_block (4 or 8 warps; default 8)
    const int wpb = plan.warps_per_block == 4 ? 4 : 8;
    // resident blocks per SM: fixed for this kernel, device and block size,
    // so queried once (a host call per run shows in short runs)
    static std::atomic<int> occupancy[64][2];
    std::atomic<int> *occ = ctx->device >= 0 && ctx->device < 64 ? &occupancy[ctx->device][wpb == 8] : nullptr;
    int per_sm = occ ? occ->load(std::memory_order_relaxed) : 0;
    if (per_sm < 1) {
        PPR_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(
            &per_sm, k_walk_persistent<E, SEG, STATS>, 32 * wpb, 0));
        if (per_sm < 1) per_sm = 1;
        if (occ) occ->store(per_sm, std::memory_order_relaxed);
    }
    int64_t blocks = (int64_t)ctx->sms * per_sm;
    int64_t needed = ((int64_t)kp.nchunks + wpb - 1) / wpb;
    if (blocks > needed) blocks = std::max<int64_t>(needed, 1);
    if ((rc = walker_event(r, st))) return rc;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)blocks);
    cfg.blockDim = dim3(32 * wpb);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    if (plan.l2_persist && ctx->l2_persist_max > 0 && ctx->l2_window_max > 0) {
        // the alias node records, or the front of the slots, persisting in L2
        constexpr bool alias = E::kAlias;
        const size_t all = alias ? (size_t)kp.n_anode * sizeof(AliasNode) : (size_t)kp.n_slots * sizeof(Sector);
        const size_t bytes = std::min(all, ctx->l2_window_max);
        if (ctx->l2_persist_set < std::min(bytes, ctx->l2_persist_max)) {
            ctx->l2_persist_set = std::min(bytes, ctx->l2_persist_max);
            PPR_CUDA(cudaDeviceSetLimit(cudaLimitPersistingL2CacheSize, ctx->l2_persist_set));
        }
        attr[0].id = cudaLaunchAttributeAccessPolicyWindow;
        attr[0].val.accessPolicyWindow.base_ptr = alias ? (void *)kp.anode : (void *)kp.slots;
        attr[0].val.accessPolicyWindow.num_bytes = bytes;
        attr[0].val.accessPolicyWindow.hitRatio = std::min(1.0f, (float)ctx->l2_persist_set / (float)bytes);
        attr[0].val.accessPolicyWindow.hitProp = cudaAccessPropertyPersisting;
        attr[0].val.accessPolicyWindow.missProp = cudaAccessPropertyStreaming;
        cfg.attrs = attr;
        cfg.numAttrs = 1;
    }
    PPR_CUDA(cudaLaunchKernelEx(&cfg, k_walk_persistent<E, SEG, STATS>, kp));
    note_launch();
    PPR_CUDA(cudaGetLastError());
    if ((rc = walker_event(r, st))) return rc;
    return launch_aggregate(ctx, AggParams{kp.ends, kp.R, kp.P2, S, kp.out_row0, kp.out, kp.order, kp.tab}, st);
}

// Chunk table of a batched graph, built on the device: chunks of at most CS
// sources that never cross an instance boundary, with positions relative to
// s_begin; the count goes to *nchunks.
__global__ void k_chunk_count(int32_t count, const int64_t *node_off, int64_t s_begin, int64_t s_end, uint32_t CS,
                              uint32_t *cnt)
{
    for (int32_t gi = blockIdx.x * blockDim.x + threadIdx.x; gi < count; gi += gridDim.x * blockDim.x) {
        const int64_t a = max(node_off[gi], s_begin), b = min(node_off[gi + 1], s_end);
        cnt[gi] = b > a ? (uint32_t)((b - a + CS - 1) / CS) : 0u;
    }
}

// One chunk a thread (with one instance a thread the largest instance's
// chunks, written one after the other, took 855 us of a 256-graph batch; now
// 11 us).
__global__ void __launch_bounds__(256) k_chunk_fill(int32_t count, const int64_t *node_off, int64_t s_begin,
                                                    int64_t s_end, uint32_t CS, const uint64_t *offs, int4 *chunks,
                                                    unsigned long long *nchunks)
{
    const uint64_t n = offs[count];
    if (blockIdx.x == 0 && threadIdx.x == 0) *nchunks = n;
    for (uint64_t c = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; c < n; c += (uint64_t)gridDim.x * blockDim.x) {
        int32_t lo = 0, hi = count;  // the instance with offs[g] <= c < offs[g + 1]
        while (hi - lo > 1) {
            const int32_t mid = (lo + hi) >> 1;
            if (offs[mid] <= c) lo = mid;
            else hi = mid;
        }
        const int64_t a = max(node_off[lo], s_begin), b = min(node_off[lo + 1], s_end);
        const int64_t s = a + (int64_t)(c - offs[lo]) * CS;
        chunks[c] = make_int4((int)(s - s_begin), (int)min((int64_t)CS, b - s), lo, (int)node_off[lo]);
    }
}

// sources per chunk, at most as many as a warp has places for; a chunk holds at
// most 2^19 walks (walk indices within a chunk stay below 2^20 for the
// multiply-shift division by R)
uint32_t chunk_sources(const RunPlan &plan)
{
    const uint32_t cs = plan.chunk_sources > 0 ? (uint32_t)plan.chunk_sources : std::max(1u, 400u / plan.R);
    return std::min(std::min(cs, kChunkSources), std::max(1u, (1u << 19) / plan.R));
}

static size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }

size_t launch_workspace_bytes(const ppr_graph *g, const RunPlan &plan, int64_t S)
{
    size_t b = align256((size_t)S * plan.R * sizeof(uint32_t));  // endpoints
    if (g->instances > 0 && plan.kernel == PPR_KERNEL_PERSISTENT) {
        const uint32_t CS = chunk_sources(plan);
        const int64_t cnt = g->instances;
        const int64_t tiles = (cnt + kScanTile - 1) / kScanTile;
        b += align256(sizeof(int4) * (size_t)((S + CS - 1) / CS + cnt + 1));  // chunk table
        b += align256(sizeof(uint32_t) * (size_t)cnt);                      // per-instance chunk counts
        b += align256(sizeof(uint64_t) * (size_t)(cnt + 1));                // their offsets
        b += align256(sizeof(uint64_t) * (size_t)(tiles + 2));              // scan scratch
    }
    return b;
}

// Every kernel a run can launch is loaded here, once per device.  With lazy
// module loading the first launch of a kernel may wait for the device to go
// idle; loaded up front, a run's launches stay asynchronous.
template <class E, bool SEG, bool STATS>
static void preload_walkers()
{
    cudaFuncAttributes a;
    cudaFuncGetAttributes(&a, k_walk_plain<E, SEG, STATS>);
    cudaFuncGetAttributes(&a, k_walk_persistent<E, SEG, STATS>);
}

void preload_run_kernels()
{
    preload_walkers<NarrowEdges, false, false>();
    preload_walkers<NarrowEdges, true, false>();
    preload_walkers<NarrowEdges, false, true>();
    preload_walkers<NarrowEdges, true, true>();
    preload_walkers<Far<NarrowEdges>, false, false>();
    preload_walkers<Far<NarrowEdges>, true, false>();
    preload_walkers<Far<AliasEdges>, false, false>();
    preload_walkers<WideEdges, false, false>();
    preload_walkers<WideEdges, true, false>();
    preload_walkers<WideEdges, false, true>();
    preload_walkers<WideEdges, true, true>();
    preload_walkers<AliasEdges, false, false>();
    preload_walkers<AliasEdges, false, true>();
    cudaFuncAttributes a;
    cudaFuncGetAttributes(&a, k_aggregate<1>);
    cudaFuncGetAttributes(&a, k_aggregate<2>);
    cudaFuncGetAttributes(&a, k_aggregate<4>);
    cudaFuncGetAttributes(&a, k_aggregate<8>);
    cudaFuncGetAttributes(&a, k_aggregate_block<128, 4>);
    cudaFuncGetAttributes(&a, k_aggregate_block<256, 4>);
    cudaFuncGetAttributes(&a, k_aggregate_block<512, 4>);
    cudaFuncGetAttributes(&a, k_aggregate_block<512, 8>);
    cudaFuncGetAttributes(&a, k_chunk_count);
    cudaFuncGetAttributes(&a, k_chunk_fill);
    cudaFuncGetAttributes(&a, k_scan_one);
    cudaFuncGetAttributes(&a, k_scan_tile_sums);
    cudaFuncGetAttributes(&a, k_scan_tile_offsets);
    cudaFuncGetAttributes(&a, k_scan_apply);
    cudaGetLastError();
}

template <class E>
static int launch_layout(ppr_ctx *ctx, const KParams &kp, const RunPlan &plan, int64_t S, cudaStream_t st,
                         ppr_result *ev_owner)
{
    if (plan.stats)
        return plan.segments ? launch_typed<E, true, true>(ctx, kp, plan, S, st, ev_owner)
                             : launch_typed<E, false, true>(ctx, kp, plan, S, st, ev_owner);
    return plan.segments ? launch_typed<E, true, false>(ctx, kp, plan, S, st, ev_owner)
                         : launch_typed<E, false, false>(ctx, kp, plan, S, st, ev_owner);
}

// The arrays a walk reads: the layout's, or those of its alias or segment tables.
void set_layout(KParams &kp, const ppr_graph *g, bool segments, bool alias)
{
    kp.tab = alias ? g->alias.tab : (segments ? g->seg.tab : g->tab);
    kp.slots = g->slots;
    kp.seg_slots = g->seg.slots;
    kp.aslots = g->alias.slots;
    kp.single = segments ? g->seg.single : g->single;
    kp.edges = g->edges;
    kp.anode = g->alias.node;
    kp.seg = g->seg.entries;
    kp.seg_head = g->seg.head;
    kp.node = g->node;
    kp.code_of = g->code_of;
    kp.order = g->order;
    kp.n_nodes = (uint64_t)g->n;
    kp.n_anode = (uint64_t)g->alias.nodes;
    kp.n_slots = (uint64_t)g->n_slots;
    kp.n_seg_slots = (uint64_t)g->seg.n_slots;
    kp.n_single = (uint64_t)g->n_single;
    kp.n_records = (uint64_t)g->m;
    kp.n_seg = (uint64_t)g->seg.entries_cap;
}

// Whether a walk's random loads are fetched by 64 bytes (Far): where the slots
// (the alias slots) are 16 times the L2 and more, a neighbour that comes along
// is evicted before it is used.  R-MAT scale 24 on two GPUs, without / with:
// job 109.05 / 105.63 and 103.57 / 103.51 ms, a quarter with segments 25.39 /
// 24.59 and 24.09 / 23.99, with alias tables 24.34 / 24.03 and 23.50 / 23.22.
// Scale 20 (three times the L2), where neighbours are used: 8.21 / 8.49 on the
// first, and alias tables 5.48 / 5.90.
static bool is_far(const ppr_ctx *ctx, const ppr_graph *g, bool alias)
{
    const double bytes = alias ? (double)g->m * sizeof(AliasRec) : (double)g->n_slots * sizeof(Sector);
    return !g->wide && g->instances == 0 &&
           (ctx->force_far < 0 ? bytes >= 16.0 * (double)ctx->l2_bytes : ctx->force_far == 1);
}

int launch_walks(ppr_ctx *ctx, const ppr_graph *g, const RunPlan &plan, const Outputs &o, int64_t s_begin, int64_t S,
                 const uint32_t *src_list, int64_t out_row0, unsigned char *ws, cudaStream_t st, ppr_result *ev_owner,
                 bool reset_queue)
{
    if (S <= 0) return PPR_OK;
    KParams kp{};
    set_layout(kp, g, plan.segments, plan.sampler == 1);
    kp.R = plan.R;
    kp.T = plan.T;
    kp.key.set((uint32_t)plan.seed, (uint32_t)(plan.seed >> 32));
    kp.tag = plan.tag;
    kp.dangling = plan.dangling;
    kp.s_begin = s_begin;
    kp.s_end = s_begin + S;
    kp.src_list = src_list;
    kp.out_row0 = out_row0;
    kp.out.nnz = o.nnz;
    kp.out.cols = o.cols;
    kp.out.cnts = o.cnts;
    kp.out.topk_idx = o.topk_idx;
    kp.out.topk_cnt = o.topk_cnt;
    kp.out.cap = o.cap;
    kp.out.topk = o.topk;
    kp.steps = o.counters;
    kp.queue = o.counters + 1;
    uint32_t P2 = 1;
    while (P2 < plan.R) P2 <<= 1;
    kp.P2 = P2;
    kp.r_magic = ((1ull << 40) + plan.R - 1) / plan.R;
    kp.refill = plan.refill_lanes > 0 ? (uint32_t)std::min(plan.refill_lanes, 32) : kDefaultRefill;
    kp.err = o.counters + 4;
    kp.ends = reinterpret_cast<uint32_t *>(ws);
    size_t off = align256((size_t)S * plan.R * sizeof(uint32_t));

    if (plan.kernel == PPR_KERNEL_PLAIN) {
        if (g->instances > 0) {
            kp.inst_off = g->d_node_off;
            kp.instances = g->instances;
        }
    } else {
        const uint32_t CS = chunk_sources(plan);
        if (g->instances > 0) {
            const int64_t cnt = g->instances;
            int4 *chunks = reinterpret_cast<int4 *>(ws + off);
            off += align256(sizeof(int4) * (size_t)((S + CS - 1) / CS + cnt + 1));
            uint32_t *ccount = reinterpret_cast<uint32_t *>(ws + off);
            off += align256(sizeof(uint32_t) * (size_t)cnt);
            uint64_t *coffs = reinterpret_cast<uint64_t *>(ws + off);
            off += align256(sizeof(uint64_t) * (size_t)(cnt + 1));
            uint64_t *ctmp = reinterpret_cast<uint64_t *>(ws + off);
            const int cb = (int)std::min<int64_t>((cnt + 255) / 256, 1024);
            k_chunk_count<<<cb, 256, 0, st>>>((int32_t)cnt, g->d_node_off, s_begin, s_begin + S, CS, ccount);
            note_launch();
            exclusive_scan_u32(ccount, cnt, coffs, ctmp, st);
            const int fb = (int)std::min<int64_t>(((S + CS - 1) / CS + cnt + 255) / 256, (int64_t)ctx->sms * 8);
            k_chunk_fill<<<fb, 256, 0, st>>>((int32_t)cnt, g->d_node_off, s_begin, s_begin + S, CS, coffs, chunks,
                                             o.counters + 3);
            note_launch();
            PPR_CUDA(cudaGetLastError());
            kp.chunks = chunks;
            kp.nchunks_dev = o.counters + 3;
            kp.nchunks = (uint32_t)((S + CS - 1) / CS + cnt);  // upper bound, for the grid size
        } else {
            // walks per chunk: CS sources' worth, smaller when that leaves warps
            // idle (a small run still spreads over every resident warp)
            const uint64_t walks = (uint64_t)S * plan.R;
            const uint64_t warps = (uint64_t)ctx->sms * 48;
            uint64_t cw = std::min<uint64_t>((uint64_t)CS * plan.R, 1u << 19);
            if ((walks + cw - 1) / cw < warps) cw = std::max<uint64_t>(32, (walks + warps - 1) / warps);
            cw = std::min<uint64_t>(cw, 1u << 19);
            kp.CW = (uint32_t)cw;
            kp.walks = walks;
            kp.nchunks = (uint32_t)((walks + cw - 1) / cw);
        }
        if (reset_queue) PPR_CUDA(cudaMemsetAsync(kp.queue, 0, sizeof(unsigned long long), st));
    }
    const bool far = is_far(ctx, g, plan.sampler == 1) && !plan.stats;
    if (far && plan.sampler == 1) return launch_typed<Far<AliasEdges>, false, false>(ctx, kp, plan, S, st, ev_owner);
    if (far && plan.segments) return launch_typed<Far<NarrowEdges>, true, false>(ctx, kp, plan, S, st, ev_owner);
    if (far) return launch_typed<Far<NarrowEdges>, false, false>(ctx, kp, plan, S, st, ev_owner);
    if (plan.sampler == 1)
        return plan.stats ? launch_typed<AliasEdges, false, true>(ctx, kp, plan, S, st, ev_owner)
                          : launch_typed<AliasEdges, false, false>(ctx, kp, plan, S, st, ev_owner);
    return g->wide ? launch_layout<WideEdges>(ctx, kp, plan, S, st, ev_owner)
                   : launch_layout<NarrowEdges>(ctx, kp, plan, S, st, ev_owner);
}

// ------------------------------------------------ allocation-free run ----
// Scratch for ppr_run_noalloc: a fixed array in device memory that exists on
// every GPU where this library's kernels are loaded, for the life of the
// process.  Layout: 256-byte header (steps, queue, sectors counters), then
// one 4-byte endpoint per walk.
constexpr size_t kNoAllocBytes = 64ull << 20;
constexpr size_t kNoAllocHeader = 256;
static __device__ __align__(256) unsigned char g_noalloc_scratch[kNoAllocBytes];

// Device addresses of g_noalloc_scratch, one per device, fetched on the first
// call for that device (the host-side symbol is only a stand-in).
static void *g_noalloc_ptr[64];
static std::mutex g_noalloc_mu;

static int noalloc_scratch(int device, unsigned char **out)
{
    if (device < 0 || device >= 64) {
        set_error("device %d out of range for the allocation-free entry point", device);
        return PPR_EINVAL;
    }
    std::lock_guard<std::mutex> lock(g_noalloc_mu);
    if (!g_noalloc_ptr[device]) {
        void *ptr = nullptr;
        cudaError_t e = cudaGetSymbolAddress(&ptr, g_noalloc_scratch);  // device is current
        if (e != cudaSuccess) return cuda_fail(e, "cudaGetSymbolAddress(scratch)");
        g_noalloc_ptr[device] = ptr;
    }
    *out = static_cast<unsigned char *>(g_noalloc_ptr[device]);
    return PPR_OK;
}

}  // namespace ppr

using namespace ppr;

extern "C" int ppr_run_noalloc(ppr_ctx *ctx, const ppr_graph *g, const ppr_run_args *a, uint32_t *nnz, int32_t *cols,
                               uint32_t *cnts, uint32_t cap, int32_t *topk_idx, uint32_t *topk_cnt)
{
    if (!ctx || !g || !a || !nnz || !cols || !cnts) {
        set_error("NULL argument");
        return PPR_EINVAL;
    }
    // the checks every run entry point shares (ranges, modes, tuning limits)
    RunPlan plan;
    int rc = check_run(g, a, 0, false, &plan);
    if (rc) return rc;
    // and those of this entry point: one persistent launch into caller buffers
    if (a->topk > 0 && (!topk_idx || !topk_cnt)) {
        set_error("topk = %d needs the top-k outputs", a->topk);
        return PPR_EINVAL;
    }
    if (a->kernel != PPR_KERNEL_PERSISTENT || a->stats != 0) {
        set_error("invalid mode for the allocation-free run (persistent kernel, no statistics)");
        return PPR_EINVAL;
    }
    if (g->instances > 0) {
        set_error("the allocation-free run takes plain graphs only");
        return PPR_ENOTSUP;
    }
    if (plan.segments && !(g->seg.T == plan.T && g->seg.tab)) {
        set_error("segment tables for this alpha are not built (a ppr_run with segments=1 builds them)");
        return PPR_ENOTSUP;
    }
    if (plan.sampler == 1 && !g->alias.tab) {
        set_error("alias sampler: needs tables built by an earlier ppr_run with sampler=1");
        return PPR_ENOTSUP;
    }
    const uint32_t need_cap = (uint32_t)std::min<int64_t>((int64_t)a->R, g->n);
    if (cap < need_cap) {
        set_error("row capacity %u < min(R, n) = %u", cap, need_cap);
        return PPR_EINVAL;
    }
    const int64_t S = a->src_end - a->src_begin;
    const size_t need = kNoAllocHeader + (size_t)S * a->R * sizeof(uint32_t);
    if (need > kNoAllocBytes) {
        set_error("allocation-free run needs %zu bytes of scratch for %lld sources x %u walks; the fixed scratch "
                  "holds %zu (at most %zu walks per call)",
                  need, (long long)S, a->R, kNoAllocBytes, (kNoAllocBytes - kNoAllocHeader) / sizeof(uint32_t));
        return PPR_ERANGE;
    }
    cudaError_t e = cudaSetDevice(ctx->device);
    if (e != cudaSuccess) return cuda_fail(e, "cudaSetDevice");
    unsigned char *scratch = nullptr;
    rc = noalloc_scratch(ctx->device, &scratch);
    if (rc) return rc;
    cudaStream_t st = (cudaStream_t)a->stream;
    // the counters must start at zero on every call; endpoints are overwritten
    e = cudaMemsetAsync(scratch, 0, kNoAllocHeader, st);
    if (e != cudaSuccess) return cuda_fail(e, "cudaMemsetAsync(scratch header)");

    plan.l2_persist = false;  // no device-limit change from the allocation-free path
    Outputs out{nnz, cols, cnts, cap, topk_idx, topk_cnt, a->topk, reinterpret_cast<unsigned long long *>(scratch)};
    return launch_walks(ctx, g, plan, out, a->src_begin, a->src_end - a->src_begin, nullptr, 0,
                        scratch + kNoAllocHeader, st, nullptr);
}
