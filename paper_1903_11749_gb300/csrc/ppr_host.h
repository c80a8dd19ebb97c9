// ppr_host.h -- host-side objects behind the C ABI (not part of the ABI).
#pragma once

#include <atomic>
#include <cstdint>
#include <mutex>
#include <string>
#include <vector>

#include <cuda_runtime.h>
#include <nvtx3/nvToolsExt.h>

#include "../../include/ppr.h"
#include "ppr_internal.cuh"

namespace ppr {

// Named range on the profiler timeline (NVTX) for the lifetime of the object.
struct Range {
    explicit Range(const char *name) { nvtxRangePushA(name); }
    ~Range() { nvtxRangePop(); }
    Range(const Range &) = delete;
    Range &operator=(const Range &) = delete;
};

void set_error(const char *fmt, ...);
void note_launch();  // counts every kernel launch of the library (ppr_kernel_launches)
int cuda_fail(cudaError_t e, const char *what);

#define PPR_CUDA(call)                                                 \
    do {                                                               \
        cudaError_t e_ = (call);                                       \
        if (e_ != cudaSuccess) return ::ppr::cuda_fail(e_, #call);     \
    } while (0)

// Stream-ordered device allocation (reports PPR_ENOMEM) and release.
int dev_alloc(void **p, size_t bytes, const char *what, cudaStream_t st);
void dev_free(void *p, cudaStream_t st);

struct AliasCache {
    ClassTab *tab = nullptr;   // class table of the alias walk: where the rows' alias slots are
    AliasNode *node = nullptr; // rows whose degree their class does not tell, by seq - first_node
    AliasRec *slots = nullptr; // one per edge of the rows of two and more
    int64_t nodes = 0;         // records at node
};

struct SegCache {
    uint32_t T = 0;               // threshold the tables were built for (0 = none)
    ClassTab *tab = nullptr;      // the class table with the small classes' slots replaced
    Sector *slots = nullptr;      // their slots, eligible nodes' pointing at their tables
    uint32_t *single = nullptr;   // single-edge nodes' targets, eligible ones marked
    SegHead *head = nullptr;      // their tables
    SegEntry *entries = nullptr;  // all tables
    int64_t n_slots = 0;
    int64_t nodes = 0, entries_n = 0;  // tables, and the entries they hold
    int64_t entries_cap = 0;           // entries allocated (tables sit at fixed slots, with gaps)
};

}  // namespace ppr

namespace ppr {
struct Server;
}

namespace ppr {
constexpr int kWords = 8;  // a run's counters
}

struct ppr_ctx {
    int device = 0;
    int sms = 0;
    ppr::Server *server = nullptr;  // serving state (ppr_serve_start)
    size_t l2_persist_max = 0;    // device limits for L2 access-policy windows
    size_t l2_window_max = 0;
    size_t l2_persist_set = 0;    // persisting set-aside this context asked for
    size_t l2_bytes = 0;          // L2 size (the layout's renumbering policy)
    size_t mem_bytes = 0;         // device memory (the layout's slot density)
    int32_t force_lam = -1, force_exact = -1, force_far = -1;  // ppr_debug_layout
    cudaStream_t copy_stream = nullptr;  // output copies of ppr_run_to_host
    std::atomic<int> refs{1};  // the caller's handle plus every live graph and result
};

namespace ppr {
// A graph or result keeps its context alive: ppr_destroy only drops the
// caller's reference, so handles may be freed in any order.
void ctx_retain(ppr_ctx *ctx);
void ctx_release(ppr_ctx *ctx);
}  // namespace ppr

struct ppr_graph {
    ppr_ctx *ctx = nullptr;
    cudaStream_t stream = nullptr;  // stream the graph was built on
    int64_t n = 0, m = 0;
    int64_t max_degree = 0, dangling = 0;
    bool wide = false;
    // the layout (ppr_internal.cuh)
    ppr::NodeRec *node = nullptr;     // [n] by seq
    void *edges = nullptr;            // EdgeN[m] or EdgeW[m] (padded to whole sectors)
    ppr::Sector *slots = nullptr;     // guide slots
    int64_t n_slots = 0;
    uint32_t *single = nullptr;       // targets of the single-edge nodes
    int64_t n_single = 0;
    ppr::ClassTab *tab = nullptr;     // device copy of htab
    ppr::ClassTab htab;
    uint32_t degree[ppr::kTabEntries];  // degree of an entry's rows, 0: not told by its class
    uint32_t lam_bits = 0;            // a range holds at most 2^lam_bits edges on average
    int32_t *order = nullptr;         // [n] caller id (within its instance) by seq
    uint32_t *code_of = nullptr;      // [n] code by caller id
    bool renumbered = false;          // what ppr_graph_info reports (the flags' rule)
    // block-diagonal instances
    int32_t instances = 0;
    std::vector<int64_t> node_off;  // host copy, count+1
    int64_t *d_node_off = nullptr;  // device copy
    ppr::SegCache seg;
    ppr::AliasCache alias;
    int64_t device_bytes = 0;
};

struct ppr_result {
    ppr_ctx *ctx = nullptr;
    const ppr_graph *g = nullptr;
    cudaStream_t stream = nullptr;
    int64_t S = 0;
    uint32_t R = 0;
    int32_t topk = 0;
    uint32_t cap = 0;
    int64_t src_begin = 0;
    uint32_t *d_nnz = nullptr;
    int32_t *d_cols = nullptr;
    uint32_t *d_cnts = nullptr;
    int32_t *d_topk_idx = nullptr;
    uint32_t *d_topk_cnt = nullptr;
    unsigned long long *d_steps = nullptr;  // counters: [0] steps, [1] work queue, [2] sectors, [3] chunks,
                                            // [4] checked-build flags, [5] flat-CSR model sectors
    cudaEvent_t ev_start = nullptr, ev_done = nullptr;
    int words = -1;                    // block of the page-locked words that the run stores its counters in
    cudaEvent_t ev_counts = nullptr;   // when it has
    void *block = nullptr;       // one allocation behind the buffers of a small run, or null
    std::vector<cudaEvent_t> walk_events;  // (before, after) each walker launch
    bool waited = false;
    uint64_t steps = 0, sectors = 0, model_sectors = 0;
    float kernel_ms = 0.f;  // walker launches only
    float run_ms = 0.f;     // walkers, reductions and everything between
    int64_t nnz_total = -1;
    std::vector<void *> scratch;  // freed with the result
};

namespace ppr {

// graph.cu
int build_graph(ppr_ctx *ctx, int64_t n, int64_t m, const int64_t *row_ptr, const int32_t *col,
                const uint32_t *w, bool device_ptrs, bool renumber, cudaStream_t st, ppr_graph *g);
// renumber.cu: numbers the nodes class by class (see ClassTab).  Fills order,
// code_of, htab (addresses counted from the arrays' starts), degree, n_single
// and n_slots; checks row_ptr.
struct LayoutStats {
    unsigned long long max_degree;
    unsigned long long dangling;
    unsigned int status;
};
enum : uint32_t { kBadRowPtr = 1u, kBadCol = 2u, kBadWeight = 4u, kWide = 8u, kBigDegree = 16u };
int number_nodes(const ppr_ctx *ctx, int64_t n, int64_t m, const int64_t *d_rp, const int64_t *d_off, uint32_t *heads,
                 LayoutStats *d_stats, bool wide, cudaStream_t st, ppr_graph *g, std::vector<void *> &tmp);
int build_segments(ppr_graph *g, uint32_t T, cudaStream_t st);
int build_alias(ppr_graph *g, cudaStream_t st);

// walk.cu
void preload_run_kernels();  // loads every kernel a run launches (once per device)

// Idle lanes before a warp starts new walks, unless the caller says: starting
// them costs the whole warp some forty instructions (256-graph batch 17.6 ms
// at one lane, 17.0 at four, 16.9 at eight, 17.9 at sixteen; the scale-24 and
// scale-20 walkers, which wait for memory, are level from one to eight).
constexpr uint32_t kDefaultRefill = 8;
struct RunPlan {
    uint32_t T, R;
    uint64_t seed;
    uint32_t tag;
    int32_t dangling;
    bool segments;
    int32_t kernel;
    int32_t warps_per_block;
    int32_t chunk_sources;
    int32_t refill_lanes;  // persistent kernel: idle lanes before a warp refills (0 = kDefaultRefill)
    bool stats;
    int32_t sampler;  // 0 first-prefix-above rule, 1 integer alias method
    bool l2_persist;  // walker launches keep the front of the layout in L2 (access-policy window)
};
// Enqueues the walks of sources [s_begin, s_end) writing output rows from
// out_row0; their S * R endpoints go to the front of the workspace.
// Where a launch writes: rows (nnz / cols / cnts at row * cap), top-k, and
// the counters block: [0] steps, [1] work queue, [2] sectors, [3] chunk count.
struct Outputs {
    uint32_t *nnz;
    int32_t *cols;
    uint32_t *cnts;
    uint32_t cap;
    int32_t *topk_idx;
    uint32_t *topk_cnt;
    int32_t topk;
    unsigned long long *counters;
};

// Argument checks shared by every run entry point (api.cu); count = number of
// sources of an explicit list (list = true), else the range is checked.
// Fills *plan; returns a PPR_* status with the message set.
int check_run(const ppr_graph *g, const ppr_run_args *a, int64_t count, bool list, RunPlan *plan);

// Sources a work chunk holds under a plan (its chunk_sources, or the library's
// choice, as far as a warp has places for them).
uint32_t chunk_sources(const RunPlan &p);

// Device workspace one launch of S sources needs (endpoints, chunk table).
size_t launch_workspace_bytes(const ppr_graph *g, const RunPlan &p, int64_t S);

// Enqueues walks and reduction for S sources: node s_begin + i, or
// src_list[i] (device) when given; rows go to out_row0 + i.  ws holds
// launch_workspace_bytes.  ev_owner: record walker-time events into it.
// The persistent walker's work queue (o.counters[1]) must be zero when the
// launch runs: callers zero the counters before their first launch and pass
// reset_queue for every later launch on the same counters.
int launch_walks(ppr_ctx *ctx, const ppr_graph *g, const RunPlan &p, const Outputs &o, int64_t s_begin, int64_t S,
                 const uint32_t *src_list, int64_t out_row0, unsigned char *ws, cudaStream_t st, ppr_result *ev_owner,
                 bool reset_queue = false);

}  // namespace ppr
