// walk_step.cuh -- one step of one walk (Sec. 2.1, Algorithm 2), shared by
// the batch walkers (walk.cu) and the serving loop (serve.cu).
//
// A step draws Philox4x32-10 at counter (s_local, j, k, tag); at a node with
// out-edges it takes the first edge whose inclusive weight prefix exceeds
// floor(r64 * W_u / 2^64) and moves to its target; at a node without
// out-edges it restarts at the source (or ends the walk, dangling mode 1);
// then it stops iff x2 < T.  At a node carrying a segment table (Algorithm 4,
// depth 3) the same draw selects one outcome: a terminated outcome ends the
// walk, an active one moves the walk and advances k by the outcome's length.
#pragma once
#include "ppr_host.h"
#include "aggregate.cuh"

namespace ppr {

struct KParams {
    const ClassTab *tab;      // the layout's class table
    const Sector *slots;      // guide slots (checked build; walks find them through the table)
    const Sector *seg_slots;  // those of the segment tables (checked build)
    const AliasRec *aslots;   // alias slots
    const uint32_t *single;   // targets of the single-edge nodes
    const void *edges;        // EdgeN / EdgeW records (ranges that overflow their slot)
    const AliasNode *anode;   // alias tables: records of the rows looked up (checked build, L2 window)
    const SegEntry *seg;      // segment tables
    const SegHead *seg_head;  // tables of single-edge nodes, by their index
    const NodeRec *node;      // by seq (statistics launches: degrees)
    RoundKeys key;            // Philox round keys of the launch's seed
    uint32_t T, R, tag;
    int32_t dangling;
    int64_t s_begin, s_end;   // sources of this launch (global ids)
    int64_t out_row0;         // output row of s_begin
    uint32_t CW;              // walks per chunk (plain graphs; a chunk may start inside a source)
    uint32_t refill;          // idle lanes before a warp starts new walks (1..32)
    uint64_t walks;           // S * R
    uint32_t nchunks;
    const unsigned long long *nchunks_dev;  // batched graphs: chunk count written on the device
    const int4 *chunks;       // batched graphs: {position, nsrc, instance, its first node}; else null
    const uint32_t *src_list; // explicit sources (position -> node id); null: s_begin + position
    const uint32_t *code_of;  // code of a caller node (the walk's start)
    const int32_t *order;     // caller id of a node by seq (endpoints)
    const int64_t *inst_off;  // batched graphs: node_off
    int32_t instances;
    AggOut out;
    uint32_t *ends;           // S * R endpoints (codes)
    unsigned long long *queue;
    unsigned long long *steps;    // [0] draws consumed, [2] layout sectors, [5] flat-CSR model sectors (statistics launch)
    uint32_t P2;              // next_pow2(R)
    uint64_t r_magic;         // ceil(2^40 / R): walk index -> source index by multiply-shift
    uint64_t n_nodes;         // checked build: nodes
    uint64_t n_anode;         // alias tables: records at anode
    uint64_t n_slots;         // checked build: guide slots
    uint64_t n_seg_slots;     // checked build: slots of the segment tables
    uint64_t n_single;        // checked build: single-edge nodes
    uint64_t n_records;       // checked build: edge records
    uint64_t n_seg;           // checked build: segment entries allocated
    unsigned long long *err;  // checked build: flags of indices that left their array
};

// The arrays a walk of graph g reads (segments, alias: those of its tables).
void set_layout(KParams &kp, const ppr_graph *g, bool segments, bool alias);

// The class table, copied into shared memory by the block.
__device__ __forceinline__ void load_tab(ClassTab &t, const ClassTab *g)
{
    for (uint32_t i = threadIdx.x; i < kTabEntries; i += blockDim.x) t.e[i] = g->e[i];
    __syncthreads();
}

// Checked build (-DPPR_CHECKED): every index a step is about to read at is
// tested against its array first; a bad one sets a flag in p.err (1 node, 2
// slot or edge record, 4 segment table, 8 endpoint slot) and ends the walk
// instead of reading, so the host reports the run as failed; nothing traps.
#ifdef PPR_CHECKED
#define PPR_CHECK(cond, flag)                                  \
    do {                                                       \
        if (!(cond)) {                                         \
            atomicOr(p.err, (unsigned long long)(flag));       \
            pend = Pending{};                                  \
            u = kDeadEnd;                                      \
            return true;                                       \
        }                                                      \
    } while (0)
constexpr uint32_t kDeadEnd = 0;
#else
#define PPR_CHECK(cond, flag) \
    do {                      \
    } while (0)
#endif

struct Tally {
    uint32_t steps = 0;
    uint32_t sectors = 0;
    uint32_t model = 0;  // the same draws on a flat CSR searched by bisection (statistics launch)
};

// 32-byte sectors a draw at a node of out-degree d costs on a flat CSR
// searched by bisection, without reuse: the row_ptr pair, max(1, ceil(log2 d) - 1)
// sectors of prefix probes (the last few probes share a sector), the col
// entry; a dangling node reads its row_ptr pair only.
__device__ __forceinline__ uint32_t flat_model_sectors(uint32_t d)
{
    if (d == 0) return 1;
    const uint32_t lg = d > 1 ? 32u - __clz(d - 1) : 0u;  // ceil(log2 d)
    return 2u + max(1u, lg > 0 ? lg - 1 : 0u);
}

// A draw over the segment table at entries [sb, sb + sn) of total mass Q.
template <bool STATS>
__device__ __forceinline__ bool seg_step(const KParams &p, uint64_t sb, uint32_t sn, uint64_t Q, const uint4 &x,
                                         uint32_t &k, uint32_t &u, Tally &tl)
{
#ifdef PPR_CHECKED
    if (sb + sn > p.n_seg) {
        atomicOr(p.err, 4ull);
        u = kDeadEnd;
        return true;
    }
#endif
    const SegTable st{p.seg};
    const uint64_t xs = mulhi64((uint64_t)x.x | ((uint64_t)x.y << 32), Q);
    const uint4 o = STATS ? search_serial_tally(st, sb, sn, xs, tl.sectors) : search_serial(st, sb, sn, xs);
    if (STATS) tl.model += 1u + (sn <= 2 ? 1u : 2u);
    ++tl.steps;
    u = o.z;
    if ((o.w >> 8) == 0) return true;
    k += o.w & 0xffu;
    return false;
}

// A draw whose range overflows its slot needs a second, dependent load.  The
// step then returns with the sector of edge records still to read pending,
// and the lane reads it in the warp's next iteration while the other lanes
// start new draws: every iteration costs one load latency, and the few lanes
// that overflow do not hold the others.
// flags = 0: none; else bit 31, the stop decision (bit 30), the first record
// of the range in the sector (bits 8..9) and the sector's bits 32..37 (0..7);
// u then holds the draw's x (the current node is not needed any more).
struct Pending {
    uint32_t flags = 0, sector = 0;
    uint32_t degree = 0;  // statistics launches only
};

// key: the walk's Philox keys, T its stop threshold (uniform over a launch of
// the batch kernels, per lane in the serving loop).
//
// One step of one walk, or the rest of one.  Returns true when the walk has
// ended, at node u.  E: NarrowEdges, WideEdges or AliasEdges, or Far of one.  STATS: count
// the 32-byte sectors read.  k counts the draws of the walk (in segment mode
// an outcome's length instead; tl.steps then counts the draws).
template <class E, bool SEG, bool STATS, class K>
__device__ __forceinline__ bool walk_step(const KParams &p, const ClassTab &tab, const K &key, uint32_t T, uint32_t src,
                                          uint32_t sctr, uint32_t j, uint32_t tag, uint32_t &k, uint32_t &u,
                                          Pending &pend, Tally &tl)
{
    const uint32_t idx = u & kIdxMask;
    const TabEntry t = tab.e[u >> kIdxBits];  // (any u: 64 entries)
    if constexpr (E::kAlias) {
        PPR_CHECK((uint64_t)t.first + idx < p.n_nodes, 1);
        // Integer alias method: slot i = floor(r*d / 2^64), y = floor(frac * W / 2^64).
        // What depends on the node alone, the record of a row that has to be
        // looked up or the target of a single edge, is loaded before the draw.
        const bool lookup = t.kind == kKindLookup, single = t.kind == kKindSingle, dang = t.kind == kKindDangling;
        if (dang && p.dangling == 1) return true;  // the walk ends here without a step
        const uint64_t at = t.addr + ((uint64_t)idx << (lookup ? 3 : 2));
        const uint2 nr = ld_pair_if<E::kFar>(reinterpret_cast<const void *>(at & ~7ull), lookup || single);
        const uint4 x = philox4x32_10(make_uint4(sctr, j, k, tag), key);
        uint32_t to = dang ? src : ((at & 4) ? nr.y : nr.x);
        if (!single && !dang) {
            const uint32_t cnt = lookup ? (nr.y >> 8) & kCountMask : t.kind;
            const AliasRec *row = lookup ? p.aslots + (((uint64_t)nr.x | ((uint64_t)nr.y << 32)) & kBeginMask)
                                         : reinterpret_cast<const AliasRec *>(t.addr) + (uint64_t)idx * cnt;
            PPR_CHECK(row >= p.aslots && row + cnt <= p.aslots + p.n_records, 2);
            const uint64_t r64 = (uint64_t)x.x | ((uint64_t)x.y << 32);
            const uint32_t i = (uint32_t)__umul64hi(r64, (uint64_t)cnt);
            const uint64_t frac = r64 * (uint64_t)cnt;
            const uint4 rec = ld_quad<E::kFar>(row + i);  // {thr, col, alias col, W}
            const uint64_t y = mulhi64_by32((uint32_t)frac, (uint32_t)(frac >> 32), rec.w);
            to = y < rec.x ? rec.y : rec.z;
        }
        if (STATS) {
            tl.sectors += (lookup ? 2 : (dang ? 0 : 1));
            tl.model += (lookup ? 2 : (dang ? 0 : 1));
        }
        u = to;
        ++k;
        return x.z < T;
    } else {
        const uint4 x = philox4x32_10(make_uint4(sctr, j, k, tag), key);
        const bool resume = !E::kWide && pend.flags != 0;
        bool stop = x.z < T;
        uint32_t next;
        uint32_t degree = 0;  // of the node drawn at (statistics)
        if (STATS) {
            degree = resume ? pend.degree : (uint32_t)(p.node[t.first + idx].word0 >> 40) & kCountMask;
            pend.degree = degree;
        }
        const SegHead *head = nullptr;
        // the range of r64 by its top c bits, among the row's ranges
        const uint32_t slot = __funnelshift_l(x.y, idx, t.kind);
        if (t.kind >= kKindSingle && !resume) {
            if (t.kind == kKindDangling) {
                if (p.dangling == 1) {  // the walk ends here without a step
                    if (STATS) tl.model += flat_model_sectors(0);  // (a flat CSR is read to know)
                    return true;
                }
                next = src;
            } else {
                PPR_CHECK(idx < p.n_single, 2);
                next = __ldg(reinterpret_cast<const uint32_t *>(t.addr) + idx);
                if (STATS) ++tl.sectors;
                if (SEG && next == kMarkSeg)
                    head = p.seg_head + (reinterpret_cast<const uint32_t *>(t.addr) - p.single) + idx;
            }
        } else {
            const Sector *at = reinterpret_cast<const Sector *>(t.addr) + slot;
            if (resume)
                at = static_cast<const Sector *>(p.edges) + ((uint64_t)pend.sector | ((uint64_t)(pend.flags & 0xffu) << 32));
            PPR_CHECK(resume ? 4 * (uint64_t)(at - static_cast<const Sector *>(p.edges)) < p.n_records
                             : (at >= p.slots && at < p.slots + p.n_slots) ||
                                   (SEG && at >= p.seg_slots && at < p.seg_slots + p.n_seg_slots),
                      2);
            const Sector s = ld_sector<E::kFar>(at);
            if (STATS) ++tl.sectors;
            if (resume) {
                next = pick_record(s, (pend.flags >> 8) & 3u, u);
                stop = (pend.flags >> 30) & 1u;
                pend.flags = 0;
            } else if (SEG && s.v[4] == kMarkSeg) {
                return seg_step<STATS>(p, (uint64_t)s.v[5] | ((uint64_t)s.v[6] << 32), s.v[7],
                                       (uint64_t)s.v[0] | ((uint64_t)s.v[1] << 32), x, k, u, tl);
            } else if constexpr (!E::kWide) {
                const uint32_t xr = (uint32_t)mulhi64_by32(x.x, x.y, s.v[0]);
                if (s.v[4] >= kMarkOverflow) {
                    uint32_t probes = 0;
                    const uint32_t a = overflow_sector(static_cast<const EdgeN *>(p.edges), s, xr, probes);
                    if (STATS) tl.sectors += probes;
                    // bits 0..7 of v4: the first sector's high bits; 8..9: the first record, in its first sector only
                    pend.sector = s.v[5] + a;
                    pend.flags = 0x80000000u | (stop ? 0x40000000u : 0u) | (s.v[4] & (a == 0 ? 0x3ffu : 0xffu));
                    if (pend.sector < a) ++pend.flags;  // carry into the high bits
                    u = xr;
                    return false;
                }
                next = pick_slot(s, xr);
            } else {
                const uint64_t W = (uint64_t)s.v[0] | ((uint64_t)s.v[1] << 32);
                const uint64_t xw = mulhi64((uint64_t)x.x | ((uint64_t)x.y << 32), W);
                if (s.v[4] >= kMarkOverflow) {
                    const WideEdges we{static_cast<const EdgeW *>(p.edges)};
                    const uint64_t lo = (uint64_t)s.v[5] | ((uint64_t)s.v[6] << 32);
                    PPR_CHECK(lo + s.v[7] <= p.n_records, 2);
                    next = WideEdges::target(STATS ? search_serial_tally(we, lo, s.v[7], xw, tl.sectors)
                                                   : search_serial(we, lo, s.v[7], xw));
                } else {
                    const uint32_t xr = (uint32_t)(xw - range_start(W, slot - (idx << t.kind), t.kind));
                    next = s.v[3] <= xr ? s.v[6] : (s.v[2] <= xr ? s.v[5] : s.v[4]);
                }
            }
        }
        if (SEG && head) {
            const SegHead h = *head;
            if (STATS) ++tl.sectors;
            return seg_step<STATS>(p, h.where & kBeginMask, (uint32_t)(h.where >> 40) & kCountMask, h.Q, x, k, u, tl);
        }
        if (STATS) tl.model += flat_model_sectors(degree);
        u = next;
        ++k;
        if (SEG) ++tl.steps;
        return stop;
    }
}

}  // namespace ppr
