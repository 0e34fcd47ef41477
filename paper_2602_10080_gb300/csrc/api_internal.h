// api_internal.h -- host-side state behind the opaque C handles.
#pragma once

#include <atomic>
#include <cstdint>
#include <cstring>
#include <mutex>
#include <vector>

#include "../../include/sssp.h"
#include "internal.h"
#include "wave.h"

namespace sssp {

// Device buffers reused across solves on one graph.
struct Workspace {
    char* ring_mem = nullptr;     // L2 rings (data, tickets, seq, cnt)
    size_t ring_bytes = 0;
    Rings rings{};
    uint32_t nrings = 0;          // bmax * shards
    bool dirty = true;            // metadata must be reset before the next solve
    int grow_shift = 0;           // capacity doublings after overflows
    Ctrl* ctrl = nullptr;
    Ctrl* host_ctrl = nullptr;    // pinned mirror
    unsigned long long* d64 = nullptr;
    size_t d64_n = 0;
    uint32_t* d32 = nullptr;
    size_t d32_n = 0;
    uint32_t* out_d = nullptr;
    size_t out_d_n = 0;
    int32_t* out_p = nullptr;
    size_t out_p_n = 0;
    int32_t* srcs = nullptr;
    size_t srcs_n = 0;
    uint32_t* pend = nullptr;     // pending marks, one per distance slot
    size_t pend_n = 0;
    unsigned long long* tl = nullptr;   // run-time sampling buffer
    size_t tl_n = 0;
    uint32_t* tide = nullptr;           // whole-grid wavefront: barrier words, then pending bits
    size_t tide_n = 0;
    uint4* tide_items = nullptr;        // hub slices of one step
    size_t tide_items_n = 0;
    uint32_t* fan = nullptr;            // multi-source: barrier words, waiting words, distance and predecessor rows
    size_t fan_n = 0;
    uint4* fan_slices = nullptr;
    size_t fan_slices_n = 0;
    cudaEvent_t ev0 = nullptr, ev1 = nullptr, ev2 = nullptr;

    int ensure_ctrl(cudaStream_t s);
    int ensure_queue(uint32_t nrings, uint32_t nch, uint32_t margin, cudaStream_t s, int sms);
    void release();
};

struct Graph {
    uint64_t uid = 0;             // unique per created graph (a handle's address may be reused)
    int device = 0;
    int sms = 1;
    int32_t n = 0;                // real vertices
    int64_t m = 0;                // real arcs
    int32_t nv = 0;               // vertices of the device layout (real + shadow)
    int64_t mv = 0;               // arcs of the device layout
    int32_t split = 0;            // arcs per shadow vertex (0 = none split)
    int32_t layout_req = 0;       // split threshold the current layout was built for
    int32_t wtype = 0;
    int32_t* row_ptr = nullptr;   // [nv + 1]
    uint2* adj = nullptr;         // [mv] (col, weight bits)
    int32_t* owner = nullptr;     // [nv - n]
    int2* span = nullptr;         // [n] (begin, end) of a real vertex's arcs in wave_adj (a hub's slices are contiguous)
    // symmetric graphs with hubs (see check_symmetry): the arcs once more for the
    // wavefront kernels, whose rows have their light arcs first (weight bits <=
    // light_w); mid[v] ends them
    bool symmetric = false;       // every arc has its reverse of equal weight (shown arc by arc)
    uint32_t light_w = 0;
    double light_share = 0.0;     // of the arcs
    uint2* wadj = nullptr;        // [m], or null
    int32_t* mid = nullptr;       // [n] (wadj)
    uint4* quads = nullptr;       // [n][2] the first four arcs of every vertex of a thin graph (see WaveParams)
    sssp_features feat{};
    sssp_config defaults{};
    sssp_config tuned{};
    bool tuned_valid = false;
    bool tuned_queues = false;    // sssp_autotune timed the tuned queue configuration faster than the wavefront
    std::atomic<bool> wide{false};   // a solve found the front too wide for one cluster
    std::atomic<bool> deep{false};   // a batch side by side gave up: too many steps
    std::atomic<int64_t> steps{0};   // the most that a single query has taken on the wavefront kernels
    // multi-query configurations from sssp_autotune_batch, per size class
    // (the number of queries rounded down to a power of two)
    struct BatchTuned {
        int32_t nq_class;
        sssp_config cfg;
        bool queues;              // timed faster than the wavefront
    };
    std::vector<BatchTuned> batch_tuned;
    sssp_stats last{};
    Workspace ws;
    std::mutex mu;
};

// Launch shape, shared-memory layout and the graph/config part of the
// kernel parameters for one instantiation; the caller fills nq, dist,
// vbits/vmask, l2 and ctrl.
struct LaunchPlan {
    KernelKey key;
    int threads = 0;
    int bps = 0;       // blocks per SM
    int grid = 0;      // sms * bps
    size_t smem = 0;
    KParams P;
};

constexpr int32_t kDefaultSplit = 1024;   // default hub split threshold (sssp_config.split_arcs = 0)

int cuda_status(cudaError_t e);
// Serving lanes per graph uid: adds delta and returns the new count.  A
// graph whose layout is in use by a lane is not relaid out.
int lane_refs(uint64_t uid, int delta);
// Uses of a graph by servers, by its uid: while one of its queries is admitted
// or running, a cancelled one's rest too, its destruction waits.
void graph_pin(uint64_t uid, int delta);
void graph_pins_wait(uint64_t uid);
// Makes the graph's layout the one for hub split threshold `split` (caller
// holds g->mu); SSSP_E_BUSY while a serving lane uses the graph.
int ensure_layout(Graph* g, int32_t split, cudaStream_t s);
// The layout (sssp_layout.cu): hubs split into shadow vertices of `split`
// arcs.  rp0 / adj0 are the validated original arrays (device); on success
// g->row_ptr / adj / owner describe the layout (rp0 / adj0 are freed, or adj0
// kept as g->wadj, when new arrays replaced them), on failure the layout is
// untouched.
int build_layout(Graph* g, int32_t* rp0, uint2* adj0, int32_t split, cudaStream_t s);
// g->span (and g->quads) for the current layout.
int fill_span(Graph* g, cudaStream_t s);
// Original arc order from a split layout: row v of rp0 from adj[src_start[v] ..].
void launch_unsplit(const Graph* g, const int32_t* src_start, const int32_t* rp0, uint2* adj0, cudaStream_t s);
// Whether the graph is symmetric, for graphs that profit (g->symmetric).
int check_symmetry(Graph* g, const int32_t* rp0, const uint2* adj0, cudaStream_t s);
sssp_config prior_config(const Graph* g);   // the feature prior (sssp_autotune.cu)
int pred_mode_for(const Graph* g);
int plan_launch(const Graph* g, const sssp_config& cfg, int pred_mode, bool mq, LaunchPlan* out,
                bool unit = false);
bool is_device_ptr(const void* p);
void resolve_auto(const Graph* g, sssp_config* c);
void batch_delta(const Graph* g, sssp_config* c, int div);   // delta / div for multi-query launches
// The library's configuration of a multi-query launch of nq queries (the
// caller's config otherwise untouched): narrower buckets, fewer active ones
// (sssp_autotune.cu).
void batch_config(const Graph* g, sssp_config* c, int32_t nq);
// Size class of a multi-query launch (nq rounded down to a power of two).
int32_t nq_class(int32_t nq);
// The batch-tuned configuration for nq queries (same size class), or null.
const sssp_config* batch_tuned_for(const Graph* g, int32_t nq);
// The batch-tuned configuration of the largest size class, or null (serving lanes).
const sssp_config* batch_tuned_largest(const Graph* g);
int validate_config(const sssp_config* c);
// Run-time sampling request (sssp_solve_sampled): host output of cap
// samples of kTimelineFields words, the period, and the count taken.
struct Sampling {
    unsigned long long* out;
    int32_t cap;
    int32_t period_us;
    int32_t* n_out;
};

// `unit`: breadth-first search (every arc counts 1; u32 levels out).
int run_queries(Graph* g, const int32_t* srcs_host, const int32_t* srcs_dev, int32_t src0, int32_t nq,
                void* dist_out, int32_t* pred_out, const sssp_config* cfg, cudaStream_t stream,
                sssp_stats* st_out, bool unit = false, const Sampling* samp = nullptr);

inline WaveGraph wave_graph(const Graph* g) {
    return WaveGraph{g->n, g->m, g->feat.avg_w, g->feat.max_deg, g->sms, g->wide.load(),
                     g->wadj && g->light_share >= 0.02 && g->light_share <= 0.4,
                     g->wadj && g->light_share >= 0.02 && g->light_share <= 0.15,
                     g->deep.load(), g->steps.load()};
}
inline void note_steps(Graph* g, int64_t steps) {
    int64_t had = g->steps.load();
    while (had < steps && !g->steps.compare_exchange_weak(had, steps)) {}
}
// The arcs that g->span numbers.
inline const uint2* wave_adj(const Graph* g) { return g->wadj ? g->wadj : g->adj; }
// The graph's part of the multi-source kernel's parameters.
struct FanParams;
void fan_graph(const Graph* g, FanParams* p);
// The wavefront kernels (sssp_wave.cu), for calls that leave the configuration
// to the library.  kWaveNotRun: the graph or the call is not for them.
// *done (or null): the first queries of the batch that are finished all the same.
constexpr int kWaveNotRun = 1;
int run_wave(Graph* g, const int32_t* srcs_host, const int32_t* srcs_dev, int32_t src0, int32_t nq, void* dist_out,
             int32_t* pred_out, cudaStream_t stream, sssp_stats* st_out, bool unit, int32_t* done = nullptr);
template <typename T>
int grow(T** p, size_t* have, size_t want) {
    if (*have >= want && *p) return SSSP_OK;
    cudaFree(*p);
    *p = nullptr;
    *have = 0;
    cudaError_t e = cudaMalloc((void**)p, (want > 1 ? want : 1) * sizeof(T));
    if (e != cudaSuccess) {
        cudaGetLastError();
        *p = nullptr;
        return SSSP_E_NOMEM;
    }
    *have = want;
    return SSSP_OK;
}

inline uint32_t __float_as_uint_host(float f) {
    uint32_t b;
    std::memcpy(&b, &f, 4);
    return b;
}

}  // namespace sssp
