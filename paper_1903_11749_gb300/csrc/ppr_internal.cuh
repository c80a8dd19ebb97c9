// ppr_internal.cuh -- device-side building blocks of libppr.so (sm_103a).
//
// Graph layout in HBM
//
// A draw at node u is a step function of its 64 random bits r: the first edge
// whose inclusive weight prefix P exceeds x = floor(r * W_u / 2^64).  The
// layout stores that function cut into 2^c equal ranges of r (the top c bits
// of r name the range): one 32-byte slot per range holds the at most four
// edges that meet the range, so a draw reads one sector whatever the degree,
// where a search tree over P reads one per level.  A range that more edges
// meet (runs of light edges) sends the draw on to the edge records.  The
// edge drawn is the one the rule names, bit for bit: only its lookup differs.
//
// Nodes are numbered class by class (class = dangling, single edge, on large
// graphs the degree up to 24, then the number of ranges 2^c), so the 32-bit code of a node is all a walk needs to
// find its slots: the top six bits select an entry of the class table (where
// the class starts and its c), the rest count nodes within the entry.  No
// node record is read on the way.
//   code   (entry << 26) | index         names a node to the walkers
//   seq    first[entry] + index          the same node in [0, n), dense
//   order[seq]: the caller's id (within its instance);  code_of[id]: its code
//   single[]   4 B per single-edge node: the code of its target
//   slots[]    32 B per range (GuideSlot layouts below)
//   EdgeN (8 B): {uint32 P, code}   -- narrow layout, every W_u < 2^32
//   EdgeW (16 B): {uint64 P, code, pad} -- wide layout; in the caller's edge order
//   NodeRec (16 B, by seq): word0 = begin (bits 0..39) | count (bits 40..62);
//     total = W_u, or the target's code for a single edge (read by the table
//     builds and the statistics, not by walks)
//   SegEntry (16 B): {uint64 cum, code, mark_len}; P / cum are inclusive
//     prefix sums within the row / table.
//
// The paper's alias tree (Algorithm 3) splits a large neighbour set so that a
// selection visits one small set per level; Lemma 1 is the analogous
// exactness argument for reading one small set of edges instead of the row.
#pragma once

#include <cstdint>
#include <cuda_runtime.h>

namespace ppr {

constexpr uint64_t kBeginMask = (1ull << 40) - 1;
constexpr uint32_t kCountMask = (1u << 23) - 1;

struct __align__(16) NodeRec {
    uint64_t word0;
    uint64_t total;
};

struct __align__(8) EdgeN {
    uint32_t P;
    int32_t col;
};

struct __align__(16) EdgeW {
    uint64_t P;
    int32_t col;
    uint32_t pad;
};

// Alias slot (integer Algorithm 1): edge j of the row is taken when the
// draw's y < thr, else its alias; both targets and the row total W (the slot
// capacity y is scaled to) are kept so that a step reads one record after
// an 8-byte node record.
struct __align__(16) AliasRec {
    uint32_t thr;
    int32_t col;
    int32_t alias_col;
    uint32_t W;
};

// Alias row of a node whose degree its class does not tell: first slot (bits
// 0..39) | degree (bits 40..62).
struct __align__(8) AliasNode {
    uint64_t word;
};

struct __align__(16) SegEntry {
    uint64_t cum;
    uint32_t node;      // code
    uint32_t mark_len;  // (active << 8) | len
};

// Segment table of a single-edge node: entries and total mass Q.
struct __align__(16) SegHead {
    uint64_t where;  // first entry (bits 0..39) | entries (bits 40..62)
    uint64_t Q;
};

__host__ __device__ inline uint64_t pack_word0(uint64_t begin, uint32_t count)
{
    return (begin & kBeginMask) | ((uint64_t)(count & kCountMask) << 40);
}

// ------------------------------------------------------------- node codes ----
// 26 index bits and up to 62 table entries name any n < 2^31 nodes: each class
// is cut into entries of 2^26 nodes.
constexpr uint32_t kIdxBits = 26;
constexpr uint32_t kIdxMask = (1u << kIdxBits) - 1;
constexpr uint32_t kTabEntries = 64;
constexpr uint32_t kMarkOverflow = 63u << kIdxBits;  // in a slot's first code: the range overflows
constexpr uint32_t kMarkSeg = 62u << kIdxBits;       // the node carries a segment table
constexpr uint32_t kKindSingle = 64, kKindDangling = 128;  // else the class's c, 0..23
constexpr uint32_t kKindLookup = 192;  // alias table: rows listed in AliasNode records (else the rows' degree)

// addr: the entry's first slot (or single target); kind: its class's c, or one
// of the above; first: seq of its first node (0xFFFFFFFF: unused entry).
struct __align__(16) TabEntry {
    uint64_t addr;
    uint32_t kind;
    uint32_t first;
};
struct ClassTab {
    TabEntry e[kTabEntries];
};

// Class of a row of d edges: 0 dangling, 1 single edge, kExact + 1 + c for 2^c
// ranges.  Plain graphs of more than kExactMin nodes class rows of up to kExact
// edges by their degree, so that alias slots are found without a record: the
// records of all nodes would not stay in L2 there, those of the longer rows (a
// tenth) do.  Alias walker without / with such classes, R-MAT, R 100, up to
// 2^20 sources: scale 18 .982 / .982 ms, 19 1.939 / 1.942, 20 4.583 / 4.500, 21
// 5.97 / 5.86, 22 7.05 / 6.78, 23 7.81 / 7.40; scale 24, 2^22 sources, 22.1 /
// 20.9.  The prefix walker and the load are level at every one of them, so the
// line could lie at 2^20.  Batches keep few classes: every class is an area of
// its own, and with 23 more the walker of 256 graphs took 25.1 ms, not 17.6.
// More than kExactNodes nodes leave no room in the table for classes by degree.
// 2^c is the smallest power of two >= d / 2^lam_bits, and a row that fits one
// slot (four edges, three in the wide layout) is one range.
constexpr uint32_t kExact = 24, kClasses = kExact + 1 + 24;
constexpr int64_t kExactMin = 1ll << 22, kExactNodes = 1ll << 30;  // 44 classes and 16 further entries of 2^26 nodes
__host__ __device__ __forceinline__ uint32_t ceil_log2(uint32_t v)
{
    if (v <= 1) return 0;
#ifdef __CUDA_ARCH__
    return 32u - __clz(v - 1);
#else
    return 32u - (uint32_t)__builtin_clz(v - 1);
#endif
}
__host__ __device__ __forceinline__ uint32_t ranges_log2(uint32_t d, uint32_t lam_bits, bool wide)
{
    return d <= (wide ? 3u : 4u) ? 0u : ceil_log2((d + (1u << lam_bits) - 1) >> lam_bits);
}
__host__ __device__ __forceinline__ uint32_t class_of_degree(uint32_t d, uint32_t lam_bits, bool wide, bool exact)
{
    return d <= 1 || (exact && d <= kExact) ? d : kExact + 1 + ranges_log2(d, lam_bits, wide);
}

__device__ __forceinline__ uint32_t seq_of(const ClassTab &t, uint32_t code)
{
    return t.e[code >> kIdxBits].first + (code & kIdxMask);
}

// ---------------------------------------------------------------- Philox ----
// Philox4x32-10 (Salmon, Moraes, Dror, Shaw, SC'11): ten rounds; each round
// takes the 32x32->64 products of counter words 0 and 2 with two fixed
// multipliers, and the new words are (hi1 ^ c1 ^ k0, lo1, hi0 ^ c3 ^ k1, lo0);
// the key advances by the golden-ratio and sqrt(3) Weyl increments between
// rounds.
constexpr uint32_t kPhiloxW0 = 0x9E3779B9u, kPhiloxW1 = 0xBB67AE85u;

// Round keys of one seed, computed on the host for a launch whose walks share
// it: ten pairs of constants where the schedule would be eighteen additions a
// draw (256-graph batch 16.9 -> 15.9 ms, scale-20 alias walker 4.73 -> 4.58).
struct RoundKeys {
    uint32_t k0[10], k1[10];
    __host__ __device__ void set(uint32_t a, uint32_t b)
    {
        for (uint32_t r = 0; r < 10; ++r) {
            k0[r] = a + r * kPhiloxW0;
            k1[r] = b + r * kPhiloxW1;
        }
    }
    __device__ __forceinline__ uint32_t a(int r) const { return k0[r]; }
    __device__ __forceinline__ uint32_t b(int r) const { return k1[r]; }
};
// The same schedule from the two key words (lanes with keys of their own).
struct LaneKeys {
    uint32_t k0, k1;
    __device__ __forceinline__ uint32_t a(int r) const { return k0 + (uint32_t)r * kPhiloxW0; }
    __device__ __forceinline__ uint32_t b(int r) const { return k1 + (uint32_t)r * kPhiloxW1; }
};

template <class K>
__device__ __forceinline__ uint4 philox4x32_10(uint4 c, const K &key)
{
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        const uint32_t m0 = 0xD2511F53u, m1 = 0xCD9E8D57u;
        const uint64_t p0 = (uint64_t)m0 * c.x, p1 = (uint64_t)m1 * c.z;
        c = make_uint4((uint32_t)(p1 >> 32) ^ c.y ^ key.a(r), (uint32_t)p1, (uint32_t)(p0 >> 32) ^ c.w ^ key.b(r),
                       (uint32_t)p0);
    }
    return c;
}

// floor(r * W / 2^64) for a 32-bit W, exactly, with two 32x32 products.
__device__ __forceinline__ uint64_t mulhi64_by32(uint32_t r_lo, uint32_t r_hi, uint32_t W)
{
    uint64_t a = (uint64_t)r_lo * W;
    uint64_t b = (uint64_t)r_hi * W + (a >> 32);
    return b >> 32;
}

__device__ __forceinline__ uint64_t mulhi64(uint64_t r, uint64_t W) { return __umul64hi(r, W); }

// ---------------------------------------------------------------- loads ----
// One 32-byte sector in a single 256-bit load (sm_100+ vector width).
// FAR: fetched from DRAM by 64 bytes, where a load of any width moves 128 by
// default (uniform 32-byte reads over 2 GB: 122.5 DRAM bytes a load, 62.6 with
// the hint, both at 51 G loads a second: it is requests that are limited).
struct Sector {
    uint32_t v[8];
};
template <bool FAR = false>
__device__ __forceinline__ Sector ld_sector(const void *p)
{
    Sector s;
    if constexpr (FAR)
        asm("ld.global.nc.L2::64B.v8.u32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
            : "=r"(s.v[0]), "=r"(s.v[1]), "=r"(s.v[2]), "=r"(s.v[3]), "=r"(s.v[4]), "=r"(s.v[5]), "=r"(s.v[6]),
              "=r"(s.v[7])
            : "l"(p));
    else
        asm("ld.global.nc.v8.u32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
            : "=r"(s.v[0]), "=r"(s.v[1]), "=r"(s.v[2]), "=r"(s.v[3]), "=r"(s.v[4]), "=r"(s.v[5]), "=r"(s.v[6]),
              "=r"(s.v[7])
            : "l"(p));
    return s;
}

// Eight bytes for the lanes with `on` set only (the others' are undefined),
// without a branch that the compiler would carry what follows into.
template <bool FAR>
__device__ __forceinline__ uint2 ld_pair_if(const void *p, bool on)
{
    uint2 v;
    if constexpr (FAR)
        asm("{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %3, 0;\n\t@q ld.global.nc.L2::64B.v2.u32 {%0,%1}, [%2];\n\t}"
            : "=r"(v.x), "=r"(v.y)
            : "l"(p), "r"((uint32_t)on));
    else
        asm("{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %3, 0;\n\t@q ld.global.nc.v2.u32 {%0,%1}, [%2];\n\t}"
            : "=r"(v.x), "=r"(v.y)
            : "l"(p), "r"((uint32_t)on));
    return v;
}

template <bool FAR>
__device__ __forceinline__ uint4 ld_quad(const void *p)
{
    if constexpr (!FAR) return __ldg(static_cast<const uint4 *>(p));
    uint4 v;
    asm("ld.global.nc.L2::64B.v4.u32 {%0,%1,%2,%3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
    return v;
}

__device__ __forceinline__ void st_sector(void *p, const Sector &s)
{
    asm volatile("st.global.v8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"l"(p), "r"(s.v[0]), "r"(s.v[1]), "r"(s.v[2]),
                 "r"(s.v[3]), "r"(s.v[4]), "r"(s.v[5]), "r"(s.v[6]), "r"(s.v[7])
                 : "memory");
}

struct NarrowEdges {
    static constexpr bool kWide = false, kFar = false, kAlias = false;
    using Edge = EdgeN;
    const EdgeN *e;
    __device__ __forceinline__ uint2 load(uint64_t i) const
    {
        return __ldg(reinterpret_cast<const uint2 *>(e) + i);
    }
    __device__ __forceinline__ static uint64_t key(uint2 v) { return v.x; }
    __device__ __forceinline__ static uint32_t target(uint2 v) { return v.y; }
    using Rec = uint2;
};

struct WideEdges {
    static constexpr bool kWide = true, kFar = false, kAlias = false;
    using Edge = EdgeW;
    const EdgeW *e;
    __device__ __forceinline__ uint4 load(uint64_t i) const
    {
        return __ldg(reinterpret_cast<const uint4 *>(e) + i);
    }
    __device__ __forceinline__ static uint64_t key(uint4 v) { return (uint64_t)v.x | ((uint64_t)v.y << 32); }
    __device__ __forceinline__ static uint32_t target(uint4 v) { return v.z; }
    using Rec = uint4;
};

// Alias tables: walked with AliasNode records and AliasRec slots.
struct AliasEdges {
    static constexpr bool kWide = false, kFar = false, kAlias = true;
};

// The same layouts walked where they lie far beyond L2 (launch_walks).
template <class E>
struct Far : E {
    static constexpr bool kFar = true;
};

// Segment entries have the same 16-byte shape as wide edges: key = cum,
// target = node, and the fourth word carries mark_len.
struct SegTable {
    const SegEntry *e;
    __device__ __forceinline__ uint4 load(uint64_t i) const
    {
        return __ldg(reinterpret_cast<const uint4 *>(e) + i);
    }
    __device__ __forceinline__ static uint64_t key(uint4 v) { return (uint64_t)v.x | ((uint64_t)v.y << 32); }
    __device__ __forceinline__ static uint32_t target(uint4 v) { return v.z; }
    using Rec = uint4;
};

// Smallest index e in [lo, lo+n) with key(e) > x, given key(lo+n-1) > x.
// Thread-serial bisection; returns the record at e.
template <class E>
__device__ __forceinline__ typename E::Rec search_serial(const E &edges, uint64_t lo, uint32_t n, uint64_t x)
{
    while (n > 1) {
        uint32_t half = n >> 1;
        typename E::Rec v = edges.load(lo + half - 1);
        if (E::key(v) <= x) {
            lo += half;
            n -= half;
        } else {
            n = half;
        }
    }
    return edges.load(lo);
}

// The same bisection, also counting the distinct 32-byte sectors its probes
// touch (consecutive probes in one sector count once).  Used by the
// statistics launch that measures the algorithmic bytes of a run.
template <class E>
__device__ __forceinline__ typename E::Rec search_serial_tally(const E &edges, uint64_t lo, uint32_t n, uint64_t x,
                                                              uint32_t &sectors)
{
    const uint64_t base = reinterpret_cast<uint64_t>(edges.e);
    constexpr uint64_t rec = sizeof(typename E::Rec);
    uint64_t last = ~0ull;
    while (n > 1) {
        uint32_t half = n >> 1;
        uint64_t sec = (base + (lo + half - 1) * rec) >> 5;
        if (sec != last) ++sectors, last = sec;
        typename E::Rec v = edges.load(lo + half - 1);
        if (E::key(v) <= x) {
            lo += half;
            n -= half;
        } else {
            n = half;
        }
    }
    uint64_t sec = (base + lo * rec) >> 5;
    if (sec != last) ++sectors;
    return edges.load(lo);
}

// ------------------------------------------------------------ guide slots ----
// The range of r with top bits b covers x in [X0, X1], X0 = floor(b W / 2^c)
// and X1 = ceil((b + 1) W / 2^c) - 1; the edges that meet it are lo .. hi, the
// first with P > X0 and the first with P > X1.
//
// Narrow slot, at most 4 edges:
//   v0 = W;  v1..v3 = P of edges lo, lo+1, lo+2;  v4..v7 = codes of lo .. lo+3
//   (missing ones repeat the last edge, so any rank past it reads the same code)
// Narrow slot, overflow: the edge records of lo .. hi lie in nsec sectors of
// four records; cut into five groups of gs = ceil(nsec / 5) sectors,
//   v0 = W;  v1..v3, v7 = last P of groups 0..3 (0xFFFFFFFF: none)
//   v4 = kMarkOverflow | (lo & 3) << 8 | first sector (bits 32..37)
//   v5 = first sector (low word);  v6 = nsec
// Wide slot, at most 3 edges (offsets from X0, which fit 32 bits since
// 2^c >= d edges of 32-bit weight):
//   v0,v1 = W;  v2,v3 = P - X0 of edges lo, lo+1;  v4..v6 = codes of lo .. lo+2
// Wide slot, overflow: v0,v1 = W;  v4 = kMarkOverflow;  v5 = lo (low word);
//   v6 = lo (high bits);  v7 = edges to search
// Node with a segment table: v0,v1 = Q;  v4 = kMarkSeg;  v5,v6 = first entry;
//   v7 = entries
constexpr uint32_t kGroups = 5;

// Code of the edge of a narrow slot that x falls on.
__device__ __forceinline__ uint32_t pick_slot(const Sector &s, uint32_t x)
{
    const uint32_t lo = s.v[1] <= x ? s.v[5] : s.v[4], hi = s.v[3] <= x ? s.v[7] : s.v[6];
    return s.v[2] <= x ? hi : lo;
}

// floor(b * W / 2^c) for b <= 2^c <= 2^23
__device__ __forceinline__ uint64_t range_start(uint64_t W, uint32_t b, uint32_t c)
{
    const uint64_t lo = W * b, hi = __umul64hi(W, (uint64_t)b);
    return c ? (hi << (64 - c)) | (lo >> c) : lo;
}

// The sector of edge records (of the whole edge array) that holds the first
// edge with P > x of a narrow overflow slot, counted from the slot's first.
__device__ __forceinline__ uint32_t overflow_sector(const EdgeN *E, const Sector &s, uint32_t x, uint32_t &probes)
{
    const uint32_t g = (s.v[1] <= x) + (s.v[2] <= x) + (s.v[3] <= x) + (s.v[7] <= x), nsec = s.v[6];
    if (nsec <= kGroups) return g;  // one sector a group
    const uint32_t gs = (nsec + kGroups - 1) / kGroups;
    const uint64_t sec0 = (uint64_t)s.v[5] | ((uint64_t)(s.v[4] & 0xffu) << 32);
    uint32_t a = g * gs, n = min(gs, nsec - a);
    while (n > 1) {
        const uint32_t half = n >> 1;
        ++probes;
        if (__ldg(&E[4 * (sec0 + a + half) - 1].P) <= x) {
            a += half;
            n -= half;
        } else {
            n = half;
        }
    }
    return a;
}

// Code of the first record i >= first of a sector of edge records with P > x
// (one of them is, by the choice of the sector).
__device__ __forceinline__ uint32_t pick_record(const Sector &r, uint32_t first, uint32_t x)
{
    const bool h0 = first == 0 && r.v[0] > x, h1 = first <= 1 && r.v[2] > x, h2 = first <= 2 && r.v[4] > x;
    return h0 ? r.v[1] : (h1 ? r.v[3] : (h2 ? r.v[5] : r.v[7]));
}

// ------------------------------------------------------------------ sort ----
// The sort of aggregate_source (aggregate.cuh), a warp's in shared memory.

__device__ __forceinline__ uint32_t next_pow2(uint32_t v)
{
    uint32_t p = 1;
    while (p < v) p <<= 1;
    return p;
}

template <class T>
__device__ __forceinline__ void warp_bitonic_sort(T *a, uint32_t n_pow2)
{
    const uint32_t lane = threadIdx.x & 31;
    for (uint32_t k = 2; k <= n_pow2; k <<= 1) {
        for (uint32_t j = k >> 1; j > 0; j >>= 1) {
            for (uint32_t i = lane; i < n_pow2; i += 32) {
                uint32_t l = i ^ j;
                if (l > i) {
                    T x = a[i], y = a[l];
                    bool up = (i & k) == 0;
                    if ((x > y) == up) {
                        a[i] = y;
                        a[l] = x;
                    }
                }
            }
            __syncwarp();
        }
    }
}

}  // namespace ppr
