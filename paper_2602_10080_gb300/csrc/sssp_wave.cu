// sssp_wave.cu -- host side of the wavefront kernels (wave.cuh): which calls
// they take, their launch shape, and one call's launch sequence.
#include <algorithm>
#include <cstring>
#include <mutex>

#include "../../include/sssp.h"
#include "api_internal.h"
#include "fan.h"
#include "wave.h"

namespace sssp {

namespace {

uint32_t pow2_at_least(double x) {
    uint32_t p = 1;
    while (p < x && p < (1u << 30)) p <<= 1;
    return p;
}

}  // namespace

// The pending bits of a cluster: four sets of a bit for every vertex, rounded
// up to a power of two.
constexpr int32_t kClusterVertices = 1 << 21;
static_assert((size_t)kClusterVertices / 2 / 16 <= kWaveMaxShared, "pending bits of 16 blocks");

// Side by side the queries advance by hops, and a step costs 20 us and more
// however few vertices wait.  G(n, m), random directed and power-law graphs take
// 15 to 42 steps; a small world of 10^6 vertices and 5 10^4 shortcuts takes 76
// (20 queries: 13.1 ms, 10.3 in turn); boxes, eight-neighbour grids and road maps
// hundreds to thousands (20 queries on a box of 100^3 vertices of degree 26: 80 ms,
// 22 in turn; on a road map of 4000^2 crossings: 8400 ms, 193 through the queues).
// On the largest graphs the arcs make up for more steps.
uint32_t deep_steps(int64_t m) { return (uint32_t)std::max<int64_t>(48, m >> 20); }

// Then the queries are taken one after the other on the whole grid, up to a
// number from which on the queue engine is faster, which works on all of them at
// once but 2 to 7 times as slowly on one.  The more arcs a step has, the busier
// the chip is with one query, and the later the line: from 10^5 arcs a step on
// there is next to none on a mesh.  ms in turn (queues), arcs a step in thousands:
//   eight-neighbour grid 1000^2, 5: 3 queries 19 (23), 4 25 (25), 6 35 (27); 2500^2,
//     12: 4 72 (79), 5 89 (83)
//   road maps of degree 2.5 with a few crossings of 14 arms, 1500^2, 2: 3 30 (36), 4
//     40 (39); 4000^2, 6: 2 75 (89), 3 109 (99)
//   small worlds of 10^6 vertices, 17: 4 11 (12), 8 21 (16); 50: 6 6.5 (7.8), 12 13
//     (11); 79: 12 8.6 (8.8), 20 14 (12); 109: 20 10 (11)
//   boxes of degree 26, whose arcs cost the queues more: 60^3, 49: 8 4.4 (14), 20 12
//     (20); 100^3, 124: 20 23 (36), 48 53 (56); 150^3, 311: 20 43 (74)
//   meshes, where a warp takes several hops a step: grid 1500 x 1450, 17: 8 44 (51),
//     12 65 (56); 2500^2, 25: 9 88 (91), 12 118 (101); 4000^2, 41: 9 169 (176), 11 205
//     (190); road maps 2000^2, 34: 12 64 (65), 20 104 (85); 1450^2, 45: 20 43 (43), 48
//     104 (76); 1500^2, 76: 20 28 (36), 48 67 (69); 4096^2, 220: 64 324 (534)
// A box of 100^3 vertices of degree 6, a mesh by its degrees with a wide front: 8
// 10 (9), 20 24 (16).
int32_t in_turn_limit(const WaveGraph& g) {
    const double deg = std::max(1.0, (double)g.m / (double)g.n);
    const bool thin = thin_graph(deg, g.max_deg);
    const int32_t most = !thin ? 24 : g.wide ? 8 : 0x7fffffff;
    const double busy = g.steps ? (double)g.m / (1e5 * (double)g.steps) : 1.0;
    if (busy >= 1.0) return most;
    return (int32_t)std::min((double)most, (thin && !g.wide ? 7.0 : deg > 12.0 && g.max_deg <= 64.0 ? 0.44 * deg : 3.55) / (1.0 - busy));
}

bool plan_wave(const WaveGraph& g, int32_t nq, int pred_mode, WavePlan* w) {
    const double deg = std::max(1.0, (double)g.m / (double)g.n);
    const bool hubs = g.max_deg > 64.0;
    // about the average weight over a quarter of the degree: of the widths
    // 1/2 to 4 times this, G(n, m) graphs run within 5% of the best at one hop
    // a step
    w->delta = 4.0 * g.avg_w / deg;
    // Threads of one cluster: one for eight vertices or 32 arcs, 1024 to
    // 16384 in 16 blocks (8 for the smallest).  GB300, us a solve at one hop a
    // step: directed 1000 vertices 8 x 128 76, 1 x 1024 82; grid 256^2 16 x 512
    // 1114, 8 x 512 1153, 1 x 1024 1800; grid 1024^2 16 x 1024 5670, 8 x 1024 8500.
    const uint32_t total =
        std::min(16384u, std::max(1024u, pow2_at_least(std::max((double)g.n / 8.0, (double)g.m / 32.0))));
    // On a mesh or a road map the front is thin and the hops are all there is
    // (few arcs a vertex, and none with many more: in a sparse random graph
    // some vertex has over twice the average).  There a warp goes on for several
    // hops a step with the vertices that it improved itself, and the threshold
    // moves as far.  us at 1, 4, 6 and 8 hops (width x4) before the quads: grid
    // 256^2 1132, 825, 797, 775; grid 1024^2 6150, 4139, 4021, 3835; road 900 x 777
    // 1893, 1378, 1414, 1404; grid 64 x 60 285, 220, -, 215; with them, at 6, 8 and
    // 12: grid 256^2 586, 577, 625; grid 1024^2 -, 2960, 3240.  Elsewhere a second hop may pay
    // (directed 60000 vertices of degree 6 174, 150 at 2, 255 at 8; G(10^4, 10^5)
    // 128, 115 at 2) but not on the smallest graphs (directed 10^4 vertices 102,
    // 114 at 2), nor with hubs (R-MAT-13 164, 189 at 2).
    const bool thin = thin_graph(deg, g.max_deg);
    const int32_t hops = thin ? 8 : !hubs && g.m > (1 << 16) ? 2 : 1;
    if (nq == 1) {
        if (g.n <= kClusterVertices && (g.m <= (1 << 19) || (thin && !g.wide))) {
            w->hops = hops;
            w->delta *= thin ? 4.0 : 1.0;
            w->log_g = total > 1024u ? 4 : 3;
            w->threads = (int)(total >> w->log_g);
            // raise the threshold while there is less than a vertex for every
            // 16 threads: grid 256^2 775 us (800 at a 32nd), grid 1024^2 3835
            // (4134; 3800 at an eighth)
            w->front = total / 16u;
            // a random graph of equal degrees looks like a mesh and has a wide
            // front, for which 16 SMs are too few: 10^6 vertices of degree 10 take
            // 1370 us here and 310 us on the whole grid; it starts over there
            if (g.m > (1 << 19)) w->wide = 24576u;
            return true;
        }
        w->kind = kWholeGrid;
        if (hubs) {
            // power law: the arcs of the core are the work.  Without them the
            // steps count on all but the largest graphs, us without (with) the
            // core's heavy arcs: R-MAT-22 565 (1786), at width 1 and a wider light
            // bound 15% slower, at 1/4 6%; R-MAT-20 255 (920); R-MAT-18 188 (378);
            // R-MAT-16 160 (303); R-MAT-19 f32 275 (626).  With a fifth of the arcs
            // light (weights up to 15) the core does not settle in time: R-MAT-21
            // 588 (556), R-MAT-18 299 (263), so it is left out above 15%
            w->core = g.core_one;
            w->delta *= g.m > (1 << 25) ? 0.5 : 1.0;
            w->front = g.m > (w->core ? 1 << 24 : 1 << 25) ? 1u : 256u;
            // a larger slice saves listing, a smaller one spreads better: R-MAT-22
            // (and BFS) 2.87 (0.90) ms with 256 arcs, 2.51 (0.79) with 512
            w->hub_deg = 512;
        } else {
            // road 4096^2, ms at 1, 3, 4, 5 and 6 hops: 9.49 (width x2), 6.13, 5.90,
            // 5.80, 5.84 (x3), 6.46 at 4 hops with a front of 16384; G(2^21, 2^25)
            // 0.79 ms at one hop, 0.81 at two, 0.83 with a front of 16384
            w->front = thin ? 32768u : 4096u;
            w->hops = thin ? 5 : 1;
            if (thin) w->delta *= 3.0;
        }
        return true;
    }
    // a batch on a small graph or a mesh: one cluster per query, as wide as the
    // queries leave room for (13 queries on grid 301 x 257: 8 blocks 1690 us,
    // 4: 1880, 1: 2130; 20 queries on grid 900 x 1000 16: 8465, 8: 5820, 4: 6030).
    // A mesh too large for that goes one by one: side by side, by hops, 20 queries
    // on grid 900 x 1000 take 167 ms.  So does any graph of many steps.
    const bool mesh = thin && !g.wide;
    if (g.n > kClusterVertices || (!mesh && (g.m > (1 << 21) || (hubs && g.m > (1 << 18))))) {
        // A group of up to 32 queries side by side costs as much as this many
        // in turn on the whole grid: R-MAT-20 6 (1.40 ms), R-MAT-18 5 (0.93 ms),
        // with all arcs 7, G(200K, 2M) 14 (2.6 ms).  Predecessors of the
        // strict-improvement rule cannot be found after the distances and stay
        // with the queues.
        // (many steps of one query may be those of its distances: whether the hops
        // are as many, side by side finds out)
        const int32_t limit = in_turn_limit(g);
        const int32_t line = g.core ? 6 : hubs ? 8 : 14;
        if ((mesh || g.deep) && nq > limit) return false;
        if (mesh || g.deep || (nq < line && (g.steps <= (int64_t)deep_steps(g.m) || nq <= limit))) w->kind = kInTurn;
        else if (pred_mode != 2 && g.n <= kFanMaxVertices) w->kind = kSideBySide;
        else return false;
        return true;
    }
    if (g.m > (1 << 21)) w->wide = 24576u;
    w->log_g = 4;
    const size_t pending = pow2_at_least((double)g.n) / 2;
    while (w->log_g > 0 && (nq << w->log_g) > g.sms && pending >> (w->log_g - 1) <= kWaveMaxShared) w->log_g--;
    w->threads = (int)std::max(128u, std::min(w->log_g ? 512u : 1024u, total >> w->log_g));
    w->front = std::max(1u, (uint32_t)(w->threads << w->log_g) / 16u);
    w->hops = hops;
    w->delta *= thin ? 4.0 : 1.0;
    return true;
}

size_t wave_params(const WavePlan& w, const WaveGraph& g, bool f32, bool unit, WaveParams* p) {
    // places: a power of two of at least n, with few bits per word on a small
    // graph, so that every thread has a word
    int bits = 0, log_t = kTideLogWords;
    while ((1ll << bits) < g.n) bits++;
    if (w.kind == kOneCluster)
        for (log_t = w.log_g; (1 << (log_t - w.log_g)) < w.threads;) log_t++;
    p->log_b = std::max(0, std::min(5, bits - log_t));
    p->mask = (uint32_t)((1ull << bits) - 1);
    p->log_g = w.log_g;
    p->words = (int32_t)std::max(1u, (1u << (bits - p->log_b)) >> p->log_g);
    p->n = g.n;
    if (unit) {
        // breadth-first: level by level; on a mesh as many levels a step as hops
        p->delta = w.hops > 2 ? (uint32_t)w.hops : kInfU32;
        p->hops = w.hops > 2 ? w.hops : 1;
    } else if (f32) p->delta = __float_as_uint_host((float)std::max(1e-30, w.delta));
    else p->delta = (uint32_t)std::min(4.0e9, std::max(1.0, w.delta));
    p->front = w.front;
    if (w.core && !unit) {
        p->core_deg = w.core_deg;
        p->arcs = g.m;
    }
    p->wide = w.wide;
    p->unit = unit ? 1 : 0;
    if (!unit) p->hops = w.hops;
    p->hub_deg = w.hub_deg;
    p->has_hubs = g.max_deg > (double)w.hub_deg;
    p->timeout_ns = 20000ull * 1000000ull;
    return w.kind == kOneCluster ? (size_t)p->words * 4 * sizeof(uint32_t) : 0;
}

uint32_t tide_slices(int64_t m, int32_t hub_deg) { return (uint32_t)(m / kTideChunk + m / hub_deg + 1); }

static size_t fan_places(int32_t n) {
    size_t places = 1;
    while (places < (size_t)n) places <<= 1;
    return places;
}

constexpr size_t kFanSyncWords = sizeof(FanSync) / sizeof(uint32_t);
static_assert(kFanSyncWords % 32 == 0, "the rows start on a 128-byte line");

size_t fan_words(int32_t n, bool pred) {
    return kFanSyncWords + std::max<size_t>(32, 2 * fan_places(n)) + 32 * (size_t)n * (pred ? 2 : 1);
}

// a row of more than kFanShort arcs is cut into slices of kFanChunk
size_t fan_slices(int32_t n, int64_t m) { return (size_t)(m / kFanChunk + m / kFanShort + 1) + (size_t)n; }

void fan_carve(uint32_t* words, uint4* slices, int32_t n, int64_t m, bool pred, FanParams* p) {
    const size_t places = fan_places(n);
    p->n = n;
    p->mask = (uint32_t)(places - 1);
    p->sync = reinterpret_cast<FanSync*>(words);
    p->wait = words + kFanSyncWords;
    p->dist = p->wait + std::max<size_t>(32, 2 * places);
    p->pred = pred ? p->dist + 32 * (size_t)n : nullptr;
    p->slices = slices;
    p->rows = slices + (m / kFanChunk + m / kFanShort + 1);
}

void fan_graph(const Graph* g, FanParams* p) {
    p->max_steps = deep_steps(g->m);
    p->span = g->span;
    p->adj = wave_adj(g);
    if (wave_graph(g).core) {
        p->mid = g->mid;
        p->light_w = g->light_w;
        p->core_deg = kFanCoreArcs;
    }
}

GridTurns& grid_turns(int device) {
    static GridTurns turns[kMaxDevices];
    return turns[device % kMaxDevices];
}

uint64_t GridTurns::take() {
    std::lock_guard<std::mutex> lk(mu_);
    return next_++;
}

bool GridTurns::mine(uint64_t place) {
    std::lock_guard<std::mutex> lk(mu_);
    return now_ == place;
}

void GridTurns::wait(uint64_t place) {
    std::unique_lock<std::mutex> lk(mu_);
    cv_.wait(lk, [&] { return now_ == place; });
}

void GridTurns::leave(uint64_t place) {
    std::lock_guard<std::mutex> lk(mu_);
    left_.insert(place);
    while (left_.erase(now_)) now_++;
    cv_.notify_all();
}

namespace {

// The batch on the multi-source kernel: groups of up to 32 queries.
int run_fan(Graph* g, const int32_t* srcs_host, const int32_t* srcs_dev, int32_t nq, uint32_t* dist_out,
            int32_t* pred_out, cudaStream_t stream) {
    Workspace& ws = g->ws;
    const size_t n = (size_t)g->n;
    int rc;
    if ((rc = grow(&ws.srcs, &ws.srcs_n, (size_t)nq))) return rc;
    cudaMemcpyAsync(ws.srcs, srcs_dev ? srcs_dev : srcs_host, sizeof(int32_t) * nq,
                    srcs_dev ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice, stream);
    // (no room for the rows: the queues need less)
    if (grow(&ws.fan, &ws.fan_n, fan_words(g->n, pred_out != nullptr))) return kWaveNotRun;
    if (grow(&ws.fan_slices, &ws.fan_slices_n, fan_slices(g->n, g->m))) return kWaveNotRun;
    FanParams P;
    std::memset(&P, 0, sizeof(P));
    fan_carve(ws.fan, ws.fan_slices, g->n, g->m, pred_out != nullptr, &P);
    fan_graph(g, &P);
    P.ctrl = ws.ctrl;
    P.timeout_ns = 20000ull * 1000000ull;
    cudaEventRecord(ws.ev1, stream);   // kernel_ms: without the allocations
    const int32_t groups = (nq + 31) / 32, per = (nq + groups - 1) / groups;
    for (int32_t q0 = 0; q0 < nq; q0 += per) {
        P.nq = std::min(per, nq - q0);
        P.srcs = ws.srcs + q0;
        cudaMemsetAsync(P.sync, 0, sizeof(FanSync), stream);
        if (launch_fan(g->wtype == SSSP_W_F32 ? 1 : 0, P, g->sms, stream) != cudaSuccess) {
            cudaGetLastError();
            return kWaveNotRun;
        }
        launch_fan_out(P.dist, g->n, P.nq, dist_out + (size_t)q0 * n, g->sms, stream);
        if (pred_out) launch_fan_out(P.pred, g->n, P.nq, (uint32_t*)pred_out + (size_t)q0 * n, g->sms, stream);
    }
    return cuda_status(cudaGetLastError());
}

}  // namespace

int run_wave(Graph* g, const int32_t* srcs_host, const int32_t* srcs_dev, int32_t src0, int32_t nq, void* dist_out,
             int32_t* pred_out, cudaStream_t stream, sssp_stats* st_out, bool unit, int32_t* done) {
    if (done) *done = 0;
    // unit weights are >= 1: the packed minimum gives the smallest-index parent
    const int pred_mode = pred_out ? (unit ? 1 : pred_mode_for(g)) : 0;
    WavePlan plan;
    const WaveGraph wg = wave_graph(g);
    if (!plan_wave(wg, nq, pred_mode, &plan)) return kWaveNotRun;
    if (cudaSetDevice(g->device) != cudaSuccess) return SSSP_E_CUDA;
    const int32_t n = g->n;
    const bool f32 = g->wtype == SSSP_W_F32 && !unit;
    const bool grid = plan.kind == kWholeGrid;
    if (plan.kind == kInTurn) {
        sssp_stats sum;
        std::memset(&sum, 0, sizeof(sum));
        auto add = [&](sssp_stats one) {
            one.kernel_ms += sum.kernel_ms;
            one.total_ms += sum.total_ms;
            one.relax_arcs += sum.relax_arcs;
            one.improved += sum.improved;
            one.rounds += sum.rounds;
            sum = one;
        };
        for (int32_t q = 0; q < nq; q++) {
            // what the queries before found out may send the others elsewhere
            WavePlan rest;
            if (q && nq - q > 1 && (!plan_wave(wave_graph(g), nq - q, pred_mode, &rest) || rest.kind != kInTurn)) {
                const size_t at = (size_t)q * (size_t)n;
                int32_t more = 0;
                sssp_stats others;
                const int rc = run_wave(g, srcs_host + q, srcs_dev ? srcs_dev + q : nullptr, 0, nq - q,
                                        (uint32_t*)dist_out + at, pred_out ? pred_out + at : nullptr, stream, &others,
                                        unit, &more);
                if (done) *done = q + more;
                if (rc) return rc;
                add(others);
                break;
            }
            sssp_stats one;
            const size_t at = (size_t)q * (size_t)n;
            const int rc = run_wave(g, nullptr, nullptr, srcs_host[q], 1, (uint32_t*)dist_out + at,
                                    pred_out ? pred_out + at : nullptr, stream, &one, unit);
            if (rc) return rc;
            add(one);
        }
        g->last = sum;
        if (st_out) *st_out = sum;
        return SSSP_OK;
    }
    WaveParams P;
    std::memset(&P, 0, sizeof(P));
    const size_t smem = wave_params(plan, wg, f32, unit, &P);
    if (smem > kWaveMaxShared) return kWaveNotRun;

    Workspace& ws = g->ws;
    int rc = ws.ensure_ctrl(stream);
    if (rc) return rc;
    const size_t cells = (size_t)nq * (size_t)n;
    const bool dist_dev = is_device_ptr(dist_out), pred_dev = pred_out && is_device_ptr(pred_out);
    uint32_t* dd = (uint32_t*)dist_out;
    int32_t* pp = pred_out;
    if (!dist_dev) {
        if ((rc = grow(&ws.out_d, &ws.out_d_n, cells))) return rc;
        dd = ws.out_d;
    }
    if (pred_out && !pred_dev) {
        if ((rc = grow(&ws.out_p, &ws.out_p_n, cells))) return rc;
        pp = ws.out_p;
    }
    GridTurn turn(g->device);
    if (plan.kind != kOneCluster) {
        // what the caller has queued on its stream is over first: it may take
        // long, or wait for another thread's solve
        if (cudaStreamQuery(stream) != cudaSuccess) {
            cudaGetLastError();
            const cudaError_t se = cudaStreamSynchronize(stream);
            if (se != cudaSuccess) return cuda_status(se);
        }
        turn.wait();
    }
    cudaMemsetAsync(ws.ctrl, 0, sizeof(Ctrl), stream);
    if (plan.kind == kSideBySide) {
        if ((rc = run_fan(g, srcs_host, srcs_dev, nq, dd, pp, stream))) return rc;
    } else {
        if (pred_mode && (rc = grow(&ws.d64, &ws.d64_n, cells))) return rc;
        if (nq > 1) {
            if ((rc = grow(&ws.srcs, &ws.srcs_n, (size_t)nq))) return rc;
            cudaMemcpyAsync(ws.srcs, srcs_dev ? srcs_dev : srcs_host, sizeof(int32_t) * nq,
                            srcs_dev ? cudaMemcpyDeviceToDevice : cudaMemcpyHostToDevice, stream);
            P.srcs = ws.srcs;
        }
        P.span = g->span;
        P.adj = wave_adj(g);
        P.quads = g->quads;
        P.pull = unit && g->symmetric;
        if (plan.core && !unit) {
            P.mid = g->mid;
            P.light_w = g->light_w;
        }
        P.src0 = src0;
        P.work = pred_mode ? (void*)ws.d64 : (void*)dd;
        P.dist_out = dd;
        P.pred_out = pp;
        P.ctrl = ws.ctrl;
        if (grid) {
            if ((rc = grow(&ws.tide, &ws.tide_n, sizeof(TideSync) / 4 + 4 * (size_t)P.words))) return rc;
            P.sync = (TideSync*)ws.tide;
            P.bits = ws.tide + sizeof(TideSync) / 4;
            if (P.has_hubs) {
                P.items_cap = tide_slices(g->m, P.hub_deg);
                if ((rc = grow(&ws.tide_items, &ws.tide_items_n, 2 * (size_t)P.items_cap))) return rc;
                P.items = ws.tide_items;
            }
            cudaMemsetAsync(ws.tide, 0, sizeof(TideSync), stream);
        }
        cudaEventRecord(ws.ev1, stream);
        const cudaError_t le = grid ? launch_tide(f32 ? 1 : 0, pred_mode, P, g->sms, plan.threads, stream)
                                    : launch_wave(f32 ? 1 : 0, pred_mode, P, nq, plan.threads, smem, stream);
        if (le != cudaSuccess) {
            // no room for the cluster or the cooperative grid on this device
            cudaGetLastError();
            return kWaveNotRun;
        }
    }
    cudaEventRecord(ws.ev2, stream);
    if (!dist_dev) cudaMemcpyAsync(dist_out, dd, cells * 4, cudaMemcpyDeviceToHost, stream);
    if (pred_out && !pred_dev) cudaMemcpyAsync(pred_out, pp, cells * 4, cudaMemcpyDeviceToHost, stream);
    cudaMemcpyAsync(ws.host_ctrl, ws.ctrl, sizeof(Ctrl), cudaMemcpyDeviceToHost, stream);
    const cudaError_t ce = cudaStreamSynchronize(stream);
    if (ce != cudaSuccess) return cuda_status(ce);
    const Ctrl& hc = *ws.host_ctrl;
    if (hc.error == kErrWide) {
        g->wide = true;
        return run_wave(g, srcs_host, srcs_dev, src0, nq, dist_out, pred_out, stream, st_out, unit, done);
    }
    if (hc.error == kErrDeep) {
        g->deep = true;
        turn.end();
        return run_wave(g, srcs_host, srcs_dev, src0, nq, dist_out, pred_out, stream, st_out, unit, done);
    }
    float ms = 0;
    cudaEventElapsedTime(&ms, ws.ev1, ws.ev2);
    sssp_stats st;
    std::memset(&st, 0, sizeof(st));
    st.kernel_ms = st.total_ms = ms;
    st.reached = st.reached_arcs = -1;
    st.relax_arcs = (int64_t)hc.stats[kStRelax];
    st.improved = (int64_t)hc.stats[kStImproved];
    st.rounds = (int64_t)hc.stats[kStIter];
    st.grid_blocks = plan.kind == kOneCluster ? nq << P.log_g : g->sms;
    st.block_threads = plan.threads;
    st.attempts = 1;
    g->last = st;
    if (st_out) *st_out = st;
    if (hc.error == kErrNone && hc.finished == nq) {
        if (nq == 1 && !unit) note_steps(g, st.rounds);
        return SSSP_OK;
    }
    return hc.error == kErrTimeout ? SSSP_E_TIMEOUT : SSSP_E_CUDA;
}

}  // namespace sssp
