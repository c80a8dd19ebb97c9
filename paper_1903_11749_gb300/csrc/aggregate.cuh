// aggregate.cuh -- endpoint aggregation of libppr.so (sm_103a): the R walk
// endpoints of each source become its sparse count row (end ids ascending,
// counts summing to R; pi_hat(s, t) = count / R, Sec. 2.2) and its top-k
// (count descending, then id ascending).  One warp per source; included by
// walk.cu, whose walker writes the endpoints this reads.
#pragma once
#include "ppr_host.h"

namespace ppr {

struct AggOut {
    uint32_t *nnz;       // [S], or null: no rows (top-k only)
    int32_t *cols;       // [S * cap], or null with cnts
    uint32_t *cnts;      // [S * cap]
    int32_t *topk_idx;   // [S * topk]
    uint32_t *topk_cnt;  // [S * topk]
    uint32_t cap;
    int32_t topk;
};

// Caller id of an endpoint the walker wrote as a node code: the layout's order
// array and the first seq of each class-table entry (shared memory), or
// neither where the endpoints are caller ids already.
struct CallerIds {
    const int32_t *order = nullptr;
    const uint32_t *first = nullptr;
    __device__ __forceinline__ uint32_t operator()(uint32_t v) const
    {
        return order ? (uint32_t)__ldg(order + (first[v >> kIdxBits] + (v & kIdxMask))) : v;
    }
};

// The serving loop's reduction for R above 128: one warp, in shared memory.
// ends: the R endpoints of one source (shared memory).  sortbuf: next_pow2(R)
// uint32 and keys: next_pow2(R) uint64 of per-warp shared scratch.  Writes
// row `out_row` of the outputs.  All 32 lanes call it.
__device__ inline void aggregate_source(const uint32_t *ends, uint32_t R, uint32_t *sortbuf, uint64_t *keys,
                                        const AggOut &o, uint64_t out_row, const CallerIds &ids = CallerIds())
{
    const uint32_t lane = threadIdx.x & 31;
    const uint32_t P2 = next_pow2(R);
    for (uint32_t i = lane; i < P2; i += 32) sortbuf[i] = i < R ? ids(ends[i]) : 0xffffffffu;
    __syncwarp();
    warp_bitonic_sort(sortbuf, P2);
    // One run per distinct endpoint.  A run is found at its last element;
    // its first element comes from a lower-bound search of the sorted buffer.
    const uint64_t rbase = out_row * o.cap;
    uint32_t nrun = 0;
    for (uint32_t base = 0; base < R; base += 32) {
        uint32_t i = base + lane;
        uint32_t v = i < R ? sortbuf[i] : 0u;
        bool tail = i < R && (i == R - 1 || sortbuf[i + 1] != v);
        uint32_t m = __ballot_sync(0xffffffffu, tail);
        if (tail) {
            uint32_t r = nrun + __popc(m & ((1u << lane) - 1));
            uint32_t lo = 0, hi = i;
            while (lo < hi) {
                uint32_t mid = (lo + hi) >> 1;
                if (sortbuf[mid] < v) lo = mid + 1;
                else hi = mid;
            }
            uint32_t c = i - lo + 1;
            if (o.cols) {
                o.cols[rbase + r] = (int32_t)v;
                o.cnts[rbase + r] = c;
            }
            if (o.topk > 0) keys[r] = ((uint64_t)(~c) << 32) | v;
        }
        nrun += __popc(m);
    }
    if (lane == 0 && o.nnz) o.nnz[out_row] = nrun;
    if (o.topk > 0) {
        uint32_t K2 = next_pow2(nrun);
        for (uint32_t i = nrun + lane; i < K2; i += 32) keys[i] = ~0ull;
        __syncwarp();
        warp_bitonic_sort(keys, K2);
        const uint64_t tb = out_row * (uint64_t)o.topk;
        for (uint32_t i = lane; i < (uint32_t)o.topk; i += 32) {
            if (i < nrun) {
                uint64_t k = keys[i];
                o.topk_idx[tb + i] = (int32_t)(uint32_t)k;
                o.topk_cnt[tb + i] = ~(uint32_t)(k >> 32);
            } else {
                o.topk_idx[tb + i] = -1;
                o.topk_cnt[tb + i] = 0;
            }
        }
    }
    __syncwarp();
}

// Ascending sort of T * I elements, element t * I + k in register k of thread
// t < T (a warp, or a block).  Bitonic network in the form whose first exchange of every level mirrors
// (i with i ^ (size - 1)), so every exchange puts the smaller element first and
// no direction is tracked: strides below I stay in the thread, below 32 I in
// the warp, longer ones (T > 32) go through sm (T * I words).
template <int T, int I>
__device__ __forceinline__ void sort_ascending(uint32_t (&v)[I], uint32_t *sm, uint32_t t)
{
    // exchange with thread t ^ x; MIRROR: the partner's elements in reverse order
    auto across = [&](uint32_t x, bool mirror) {
        const bool lower = (t & (mirror ? (x + 1) >> 1 : x)) == 0;
        uint32_t o[I];
        if (T == 32 || x < 32) {
#pragma unroll
            for (int k = 0; k < I; ++k) o[k] = __shfl_xor_sync(0xffffffffu, v[mirror ? I - 1 - k : k], x);
        } else {
#pragma unroll
            for (int k = 0; k < I; ++k) sm[k * T + t] = v[k];
            __syncthreads();
#pragma unroll
            for (int k = 0; k < I; ++k) o[k] = sm[(mirror ? I - 1 - k : k) * T + (t ^ x)];
            __syncthreads();
        }
#pragma unroll
        for (int k = 0; k < I; ++k) v[k] = lower ? min(v[k], o[k]) : max(v[k], o[k]);
    };
    auto within = [&](int a, int b) {
        const uint32_t x = v[a], y = v[b];
        v[a] = min(x, y);
        v[b] = max(x, y);
    };
#pragma unroll
    for (int size = 2; size <= T * I; size <<= 1) {
        if (size <= I) {
#pragma unroll
            for (int k = 0; k < I; ++k)
                if ((k ^ (size - 1)) > k) within(k, k ^ (size - 1));
        } else {
            across(size / I - 1, true);
        }
#pragma unroll
        for (int stride = size >> 2; stride > 0; stride >>= 1) {
            if (stride < I) {
#pragma unroll
                for (int k = 0; k < I; ++k)
                    if ((k ^ stride) > k) within(k, k ^ stride);
            } else {
                across(stride / I, false);
            }
        }
    }
}

// Top-K of one row without sorting every run, for K <= 32 and more than 32 runs
// met twice or more:
// kv holds the key (R - count) << 12 | run at each run's head element, v its
// node id (kv 0xFFFFFFFF elsewhere; elements e * 32 + lane in order), and the
// answer is the K smallest keys in ascending order.  The
// count rank q = key >> 12 of the K-th smallest key is found by bisection
// over [0, R - 2] with ballot counts; every key with q below it is taken (fewer
// than K, sorted in one register per lane), then the first keys with q equal
// to it in run order (= ascending key, as runs are numbered in id order)
// fill the remaining places.  cbuf: 32 uint32 of per-warp shared memory.
template <int E>
__device__ __forceinline__ void topk_select_reg(const uint32_t (&kv)[E], const uint32_t (&v)[E], uint32_t K, uint32_t R,
                                                const uint32_t *run_id, uint32_t *cbuf, const AggOut &o, uint64_t tb)
{
    const uint32_t lane = threadIdx.x & 31, below = (1u << lane) - 1;
    auto count_le = [&](uint32_t t) {
        uint32_t c = 0;
#pragma unroll
        for (int e = 0; e < E; ++e) c += __popc(__ballot_sync(0xffffffffu, (kv[e] >> 12) <= t));
        return c;
    };
    // smallest t with count_le(t) >= K; count_le(R - 2) > 32 >= K here
    uint32_t lo = 0, hi = R - 2;
    while (lo < hi) {
        const uint32_t mid = (lo + hi) >> 1;
        if (count_le(mid) >= K) hi = mid;
        else lo = mid + 1;
    }
    const uint32_t t = lo;
    uint32_t nlt = 0;  // keys below t, gathered into cbuf in run order
#pragma unroll
    for (int e = 0; e < E; ++e) {
        const bool lt = (kv[e] >> 12) < t;
        const uint32_t ml = __ballot_sync(0xffffffffu, lt);
        if (lt) cbuf[nlt + __popc(ml & below)] = kv[e];
        nlt += __popc(ml);
    }
    __syncwarp();
    // nlt < K places for the keys below t, sorted; then K - nlt keys equal to t
    uint32_t x[1] = {lane < nlt ? cbuf[lane] : 0xffffffffu};
    sort_ascending<32, 1>(x, nullptr, lane);
    if (lane < nlt) {
        o.topk_idx[tb + lane] = (int32_t)run_id[x[0] & 0xfffu];
        o.topk_cnt[tb + lane] = R - (x[0] >> 12);
    }
    uint32_t seen = 0;
#pragma unroll
    for (int e = 0; e < E; ++e) {
        const bool eq = (kv[e] >> 12) == t;
        const uint32_t me = __ballot_sync(0xffffffffu, eq);
        const uint32_t pos = nlt + seen + __popc(me & below);
        if (eq && pos < K) {
            o.topk_idx[tb + pos] = (int32_t)v[e];
            o.topk_cnt[tb + pos] = R - t;
        }
        seen += __popc(me);
    }
}

// Top-K of a row in which nm <= 32 runs are met twice or more (most rows; all
// of them when R <= 65): runs met once come last (count 1 is the smallest) and
// already in run order, so only the nm others are sorted, in one register a
// lane, and the rest are placed by their run index less the others before
// them.  kv, v as above; many: ballots of the elements whose runs are met twice
// or more.
template <int E>
__device__ __forceinline__ void topk_ones_reg(const uint32_t (&kv)[E], const uint32_t (&v)[E], const uint32_t (&many)[E],
                                              uint32_t nm, uint32_t nrun, uint32_t K, uint32_t R, const uint32_t *run_id,
                                              uint32_t *cbuf, const AggOut &o, uint64_t tb)
{
    const uint32_t lane = threadIdx.x & 31, below = (1u << lane) - 1;
    uint32_t seen = 0;
#pragma unroll
    for (int e = 0; e < E; ++e) {
        const uint32_t before = seen + __popc(many[e] & below);
        if ((many[e] >> lane) & 1u) {
            cbuf[before] = kv[e];
        } else if (kv[e] != 0xffffffffu) {
            const uint32_t pos = nm + (kv[e] & 0xfffu) - before;
            if (pos < K) {
                o.topk_idx[tb + pos] = (int32_t)v[e];
                o.topk_cnt[tb + pos] = 1;
            }
        }
        seen += __popc(many[e]);
    }
    __syncwarp();
    uint32_t x[1] = {lane < nm ? cbuf[lane] : 0xffffffffu};
    if (nm > 1) sort_ascending<32, 1>(x, nullptr, lane);
    if (lane < nm && lane < K) {
        o.topk_idx[tb + lane] = (int32_t)run_id[x[0] & 0xfffu];
        o.topk_cnt[tb + lane] = R - (x[0] >> 12);
    }
    for (uint32_t i = nrun + lane; i < K; i += 32) {
        o.topk_idx[tb + i] = -1;
        o.topk_cnt[tb + i] = 0;
    }
}

// Register-resident variant for next_pow2(R) = 32 * E <= 256 (R <= 32: E = 1).
// The sort works on consecutive elements of a lane (its short strides are then
// plain min and max, and of the 28 stages of R = 128 only 15 are shuffles); what
// follows takes them in striped order (element e * 32 + lane in register e),
// where ballots see them in order and rows are written in whole sectors.  Runs
// are found from neighbour values; the top-k sorts 32-bit keys
// (R - count) << 12 | run, whose order is count descending then end id
// ascending because runs are numbered in id order.
// scratch: 32 * E + 32 uint32 of per-warp shared memory, 16-byte aligned.
//
// Bound by the ALU pipe, so what follows the sort is kept short: run heads
// come from one shuffle and one ballot per register; a run's count is the
// distance to the next head, read off the same ballots; and the top-k keys
// stay at their heads (0xFFFFFFFF elsewhere), so a selected run has its node
// id in the lane that holds its key.  Reductions with the chip full, ms, against
// a sort in striped order with the top-k's ties found by a second pass of
// ballots: R 50, top-64 .178 -> .156; R 100, top-32 .275 -> .232 (2^18 sources
// each); R 200 .331 -> .267 (167,772 sources).
template <int E>
__device__ inline void aggregate_source_reg(const uint32_t *ends, uint32_t R, uint32_t *scratch, const AggOut &o,
                                            uint64_t out_row, const CallerIds &ids = CallerIds())
{
    const uint32_t lane = threadIdx.x & 31;
    uint32_t *run_id = scratch, *cbuf = scratch + 32 * E;
    uint32_t v[E];
#pragma unroll
    for (int e = 0; e < E; ++e) {
        const uint32_t i = (uint32_t)e * 32 + lane;
        v[e] = i < R ? ends[i] : 0xffffffffu;
    }
    const uint64_t rbase = out_row * o.cap;
    // A row whose R endpoints are all one node (a dangling source, whose walks
    // restart where they began: 4-6 % of the sources of the R-MAT graphs) is
    // one run of count R; it skips the sort.
    const uint32_t v0 = __shfl_sync(0xffffffffu, v[0], 0);
    bool same = true;
#pragma unroll
    for (int e = 0; e < E; ++e) same = same && ((uint32_t)e * 32 + lane >= R || v[e] == v0);
    if (__all_sync(0xffffffffu, same)) {
        const int32_t id = (int32_t)ids(v0);
        if (lane == 0) {
            if (o.cols) {
                o.cols[rbase] = id;
                o.cnts[rbase] = R;
            }
            if (o.nnz) o.nnz[out_row] = 1;
        }
        const uint64_t tb = out_row * (uint64_t)o.topk;
        for (uint32_t i = lane; i < (uint32_t)max(o.topk, 0); i += 32) {
            o.topk_idx[tb + i] = i == 0 ? id : -1;
            o.topk_cnt[tb + i] = i == 0 ? R : 0u;
        }
        __syncwarp();
        return;
    }
#pragma unroll
    for (int e = 0; e < E; ++e)
        if ((uint32_t)e * 32 + lane < R) v[e] = ids(v[e]);
    sort_ascending<32, E>(v, nullptr, lane);
    if (E > 1) {  // consecutive to striped
        if constexpr (E == 2) {
            reinterpret_cast<uint2 *>(scratch)[lane] = make_uint2(v[0], v[1]);
        } else if constexpr (E >= 4) {
#pragma unroll
            for (int e = 0; e < E; e += 4)
                reinterpret_cast<uint4 *>(scratch)[(lane * E + e) / 4] = make_uint4(v[e], v[e + 1], v[e + 2], v[e + 3]);
        }
        __syncwarp();
#pragma unroll
        for (int e = 0; e < E; ++e) v[e] = scratch[e * 32 + lane];
        __syncwarp();
    }
    uint32_t hb[E], nxt[E];  // heads of each register; first head in a later register (R: none)
#pragma unroll
    for (int e = 0; e < E; ++e) {
        // the element before: lane 31 hands lane 0 the last one of the register before
        const uint32_t mine = e > 0 && lane == 31 ? v[e > 0 ? e - 1 : 0] : v[e];
        const uint32_t prev = __shfl_sync(0xffffffffu, mine, (lane + 31) & 31);
        const bool head = (uint32_t)e * 32 + lane < R && ((e == 0 && lane == 0) || prev != v[e]);
        hb[e] = __ballot_sync(0xffffffffu, head);
    }
    uint32_t after = R;
#pragma unroll
    for (int e = E - 1; e >= 0; --e) {
        nxt[e] = after;
        if (hb[e]) after = (uint32_t)e * 32 + __ffs(hb[e]) - 1;
    }
    uint32_t nrun = 0, kv[E];
#pragma unroll
    for (int e = 0; e < E; ++e) {
        kv[e] = 0xffffffffu;
        if ((hb[e] >> lane) & 1u) {
            const uint32_t i = (uint32_t)e * 32 + lane, above = hb[e] & (0xfffffffeu << lane);
            const uint32_t run = nrun + __popc(hb[e] & ((1u << lane) - 1));
            const uint32_t c = (above ? (uint32_t)e * 32 + __ffs(above) - 1 : nxt[e]) - i;
            if (o.cols) {
                o.cols[rbase + run] = (int32_t)v[e];
                o.cnts[rbase + run] = c;
            }
            run_id[run] = v[e];
            kv[e] = ((R - c) << 12) | run;
        }
        nrun += __popc(hb[e]);
    }
    if (lane == 0 && o.nnz) o.nnz[out_row] = nrun;
    if (o.topk > 0) {
        __syncwarp();
        const uint64_t tb = out_row * (uint64_t)o.topk;
        const uint32_t K = (uint32_t)o.topk;
        uint32_t many[E], nm = E > 1 ? 0 : 33;  // (one register: the whole row is sorted at once)
#pragma unroll
        for (int e = 0; e < (E > 1 ? E : 0); ++e) {
            many[e] = __ballot_sync(0xffffffffu, kv[e] < (R - 1) << 12);
            nm += __popc(many[e]);
        }
        if (nm <= 32) {
            topk_ones_reg<E>(kv, v, many, nm, nrun, K, R, run_id, cbuf, o, tb);
        } else if (E > 1 && K <= 32 && K < nrun) {
            topk_select_reg<E>(kv, v, K, R, run_id, cbuf, o, tb);
        } else {
            sort_ascending<32, E>(kv, nullptr, lane);
#pragma unroll
            for (int e = 0; e < E; ++e) {
                const uint32_t i = lane * E + e;
                if (i < K) {
                    if (i < nrun) {
                        o.topk_idx[tb + i] = (int32_t)run_id[kv[e] & 0xfffu];
                        o.topk_cnt[tb + i] = R - (kv[e] >> 12);
                    } else {
                        o.topk_idx[tb + i] = -1;
                        o.topk_cnt[tb + i] = 0;
                    }
                }
            }
            // k may exceed the sorted block (k > next_pow2(R) >= nnz): pad the rest
            for (uint32_t i = 32u * E + lane; i < K; i += 32) {
                o.topk_idx[tb + i] = -1;
                o.topk_cnt[tb + i] = 0;
            }
        }
    }
    __syncwarp();
}

// ------------------------------------------------ one block per source ----
// R > 256: a block of T threads reduces one source, I elements a thread
// (T * I = next_pow2(R)).  One warp a source left the chip idle where there
// are few sources (rankings over some hundred sources with R in the
// thousands) and waited through a chain of shared-memory or 32-register
// stages.  Reduction of 500 sources, R 4096, top-1000: 1262 -> 40 us; 1,000
// sources, R 1000: 46 -> 18 us; and with the chip full, 2^25 walks in all: R
// 300 .697 -> .505 ms, 500 .478 -> .324, 1000 .728 -> .392, 2000 7.80 -> .504,
// 4000 17.5 -> .497.

// Exclusive sum over the block's threads; *total: of all.  s: T / 32 words.
template <int T>
__device__ __forceinline__ uint32_t block_sum_before(uint32_t x, uint32_t *s, uint32_t *total)
{
    const uint32_t lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    uint32_t y = x;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t z = __shfl_up_sync(0xffffffffu, y, o);
        if (lane >= (uint32_t)o) y += z;
    }
    if (lane == 31) s[wid] = y;
    __syncthreads();
    uint32_t before = 0, all = 0;
#pragma unroll
    for (uint32_t w = 0; w < T / 32; ++w) {
        if (w == wid) before = all;
        all += s[w];
    }
    __syncthreads();
    *total = all;
    return before + y - x;
}

template <int T, int I>
struct BlockScratch {
    uint32_t id[T * I];         // sort exchange, then the runs' node ids
    uint32_t start[T * I + 1];  // first element of each run
    uint32_t key[T * I / 2];    // sort exchange of the runs met twice or more (R / 2 of them at most), then their keys
    uint32_t sums[T / 32];
    uint32_t edge[T / 32];      // last element of each warp
};

template <int T, int I>
__device__ void aggregate_source_block(const uint32_t *ends, uint32_t R, BlockScratch<T, I> &sm, const AggOut &o,
                                       uint64_t out_row, const CallerIds &ids)
{
    const uint32_t t = threadIdx.x, lane = t & 31, wid = t >> 5;
    uint32_t v[I];
#pragma unroll
    for (int k = 0; k < I; ++k) {
        const uint32_t i = (uint32_t)k * T + t;
        v[k] = i < R ? ids(ends[i]) : 0xffffffffu;
    }
    sort_ascending<T, I>(v, sm.id, t);
    if (lane == 31) sm.edge[wid] = v[I - 1];
    __syncthreads();
    uint32_t prev = __shfl_up_sync(0xffffffffu, v[I - 1], 1);
    if (lane == 0) prev = wid > 0 ? sm.edge[wid - 1] : 0u;
    uint32_t heads = 0;
#pragma unroll
    for (int k = 0; k < I; ++k) {
        const uint32_t i = t * I + k;
        if (i < R && (i == 0 || v[k] != (k > 0 ? v[k > 0 ? k - 1 : 0] : prev))) heads |= 1u << k;
    }
    uint32_t nrun;
    uint32_t run = block_sum_before<T>(__popc(heads), sm.sums, &nrun);
#pragma unroll
    for (int k = 0; k < I; ++k)
        if ((heads >> k) & 1u) {
            sm.id[run] = v[k];
            sm.start[run++] = t * I + k;
        }
    if (t == 0) {
        sm.start[nrun] = R;
        if (o.nnz) o.nnz[out_row] = nrun;
    }
    __syncthreads();
    if (o.cols) {
        const uint64_t rbase = out_row * o.cap;
        for (uint32_t r = t; r < nrun; r += T) {
            o.cols[rbase + r] = (int32_t)sm.id[r];
            o.cnts[rbase + r] = sm.start[r + 1] - sm.start[r];
        }
    }
    if (o.topk > 0) {
        const uint32_t K = (uint32_t)o.topk;
        const uint64_t tb = out_row * (uint64_t)o.topk;
        // runs met once come last, in id order, and need no sort
        uint32_t c[I], many = 0, nm;
#pragma unroll
        for (int k = 0; k < I; ++k) {
            const uint32_t r = t * I + k;
            c[k] = r < nrun ? sm.start[r + 1] - sm.start[r] : 0u;
            many += c[k] >= 2;
        }
        uint32_t mb = block_sum_before<T>(many, sm.sums, &nm);
#pragma unroll
        for (int k = 0; k < I; ++k) {
            const uint32_t r = t * I + k;
            if (c[k] >= 2) {
                sm.key[mb++] = ((R - c[k]) << 12) | r;
            } else if (c[k] == 1 && nm + r - mb < K) {
                o.topk_idx[tb + nm + r - mb] = (int32_t)sm.id[r];
                o.topk_cnt[tb + nm + r - mb] = 1;
            }
        }
        __syncthreads();
        auto put = [&](uint32_t i, uint32_t key) {
            if (i < nm && i < K) {
                o.topk_idx[tb + i] = (int32_t)sm.id[key & 0xfffu];
                o.topk_cnt[tb + i] = R - (key >> 12);
            }
        };
        if (nm <= T) {
            uint32_t x[1] = {t < nm ? sm.key[t] : 0xffffffffu};
            __syncthreads();
            sort_ascending<T, 1>(x, sm.key, t);
            put(t, x[0]);
        } else {
            uint32_t x[I / 2];
#pragma unroll
            for (int k = 0; k < I / 2; ++k) x[k] = (uint32_t)k * T + t < nm ? sm.key[k * T + t] : 0xffffffffu;
            __syncthreads();
            sort_ascending<T, I / 2>(x, sm.key, t);
#pragma unroll
            for (int k = 0; k < I / 2; ++k) put(t * (I / 2) + k, x[k]);
        }
        for (uint32_t i = nrun + t; i < K; i += T) {
            o.topk_idx[tb + i] = -1;
            o.topk_cnt[tb + i] = 0;
        }
    }
    __syncthreads();
}

// Launch parameters of k_aggregate: S sources, R endpoints each, source-major.
struct AggParams {
    const uint32_t *ends;
    uint32_t R, P2;     // P2 = next_pow2(R)
    int64_t S;
    int64_t out_row0;   // output row of the first source
    AggOut out;
    const int32_t *order;  // caller id by seq
    const ClassTab *tab;
};

// The first seq of each class-table entry, for CallerIds.
__device__ __forceinline__ CallerIds load_ids(uint32_t *first, const AggParams &p)
{
    for (uint32_t i = threadIdx.x; i < kTabEntries; i += blockDim.x) first[i] = p.tab->e[i].first;
    __syncthreads();
    return CallerIds{p.order, first};
}

// One warp per source, next_pow2(R) = 32 * E <= 256 (R <= 32: E = 1).
constexpr int kAggWarps = 4;
template <int E>
__global__ void __launch_bounds__(32 * kAggWarps) k_aggregate(AggParams p)
{
    __shared__ uint32_t first[kTabEntries];
    __shared__ __align__(16) uint32_t scratch[kAggWarps][32 * E + 32];
    const CallerIds ids = load_ids(first, p);
    const uint32_t wid = threadIdx.x >> 5;
    const uint64_t S = (uint64_t)p.S;
    for (uint64_t i = (uint64_t)blockIdx.x * kAggWarps + wid; i < S; i += (uint64_t)gridDim.x * kAggWarps)
        aggregate_source_reg<E>(p.ends + i * p.R, p.R, scratch[wid], p.out, (uint64_t)p.out_row0 + i, ids);
}

template <int T, int I>
__global__ void __launch_bounds__(T) k_aggregate_block(AggParams p)
{
    __shared__ uint32_t first[kTabEntries];
    __shared__ BlockScratch<T, I> sm;
    const CallerIds ids = load_ids(first, p);
    for (uint64_t i = blockIdx.x; i < (uint64_t)p.S; i += gridDim.x)
        aggregate_source_block<T, I>(p.ends + i * p.R, p.R, sm, p.out, (uint64_t)p.out_row0 + i, ids);
}

template <int E>
static int launch_aggregate_e(ppr_ctx *ctx, const AggParams &ap, cudaStream_t st)
{
    // 128 blocks a SM, some ten times what is resident: sixteen left a second wave
    // of a few blocks (R 50, 2^22 sources: 2.37 -> 1.98 ms; R 100, 2^20: .889 ->
    // .796; R 200, 2^21: 3.19 -> 2.94; as many as are resident .97 ms at R 100,
    // 512 a SM .81)
    const int blocks = (int)std::max<int64_t>(1, std::min<int64_t>((ap.S + kAggWarps - 1) / kAggWarps, (int64_t)ctx->sms * 128));
    k_aggregate<E><<<blocks, 32 * kAggWarps, 0, st>>>(ap);
    note_launch();
    PPR_CUDA(cudaGetLastError());
    return PPR_OK;
}

template <int T, int I>
static int launch_aggregate_block(ppr_ctx *ctx, const AggParams &ap, cudaStream_t st)
{
    // many times what is resident, as above (R 300, 1000, 4000 of 2^16, 2^15, 2^13
    // sources: 275, 344, 430 us; with an eighth of the blocks 291, 368, 462)
    const int blocks = (int)std::max<int64_t>(1, std::min<int64_t>(ap.S, (int64_t)ctx->sms * (32768 / T)));
    k_aggregate_block<T, I><<<blocks, T, 0, st>>>(ap);
    note_launch();
    PPR_CUDA(cudaGetLastError());
    return PPR_OK;
}

static int launch_aggregate(ppr_ctx *ctx, const AggParams &ap, cudaStream_t st)
{
    switch (ap.P2) {
    case 1: case 2: case 4: case 8: case 16: case 32: return launch_aggregate_e<1>(ctx, ap, st);
    case 64: return launch_aggregate_e<2>(ctx, ap, st);
    case 128: return launch_aggregate_e<4>(ctx, ap, st);
    case 256: return launch_aggregate_e<8>(ctx, ap, st);
    case 512: return launch_aggregate_block<128, 4>(ctx, ap, st);
    case 1024: return launch_aggregate_block<256, 4>(ctx, ap, st);
    case 2048: return launch_aggregate_block<512, 4>(ctx, ap, st);
    default: return launch_aggregate_block<512, 8>(ctx, ap, st);  // R <= 4096
    }
}

}  // namespace ppr
