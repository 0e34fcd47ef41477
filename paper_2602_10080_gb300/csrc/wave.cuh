// wave.cuh -- step-synchronous wavefront searches.
//
// A search is advanced in steps: the vertices that wait for relaxation are
// bits, a step relaxes them all, and a barrier ends it.  A push is one OR
// without an answer, a pop is a word, no queue can overflow, and no element
// is stale or queued twice.  Two kernels share the relaxation:
//
//   wave_kernel  one cluster of 1 to 16 blocks per query, its bits in the
//                cluster's shared memory, the hardware cluster barrier between
//                steps.  For graphs whose wavefront is thin (meshes, small
//                graphs), where the latency of a hop is all there is; a batch
//                is one cluster per query, and no cluster waits for another.
//   tide_kernel  the whole grid on one query, its bits in global memory, a
//                grid barrier between steps.  For large graphs.
//
// Order: vertices below the threshold T wait in `near` and are relaxed in the
// next step; the others wait in `far`.  When fewer than `front` vertices are
// waiting in near, T grows by delta and the far bits below it are relaxed in
// the same step (delta-stepping with a width that follows the parallelism:
// a step costs the same for one vertex and for one per thread, so a thin
// front is filled up with speculative work, which saves steps).  Every
// label-correcting order ends in the same distances.
//
// GB300, through the queues -> here: grid 256^2 with predecessors 3.13 -> 0.60 ms
// (49 steps of 8 hops), grid 1024^2 15.2 -> 2.87, 1000 vertices 236 -> 54 us; road
// 4096^2 18.1 -> 5.85 ms, G(2^21, 2^25) f32 9.7 -> 0.76, R-MAT-22 3.05 -> 0.55,
// breadth-first on it 2.12 -> 0.34.  wave_kernel is bound by the chain of a hop
// (two trips to L2, 460 + 540 cycles, and 400 to 950 of instructions between
// them), tide_kernel by steps: two thirds of its stalls are the barriers of the
// block and the grid, L2 and L1 run at 20 to 40%, DRAM at 4% (R-MAT-20) to 25%
// (R-MAT-22) of its rate.
#pragma once

#include "mlmq.cuh"

namespace sssp {

constexpr int kWaveMaxCluster = 16;
constexpr int kWaveHubs = 128;        // hubs one block expands together per step (later ones: by their warp)
constexpr uint32_t kWaveHash = 0x9E3779B1u;      // odd: v -> v * hash mod 2^bits is one to one
constexpr uint32_t kWaveHashInv = 0x0E8B2F51u;   // its inverse mod 2^32
static_assert((uint32_t)(0x9E3779B1ull * 0x0E8B2F51ull) == 1u, "inverse of the vertex hash");
constexpr uint32_t kTideChunk = 256;  // arcs of a hub that one warp relaxes at a time

struct WaveParams {
    const int2* span;         // [n] arcs of a vertex: adj[span.x .. span.y); null: from row
    const int32_t* row;       // [n + 1] row offsets (span null)
    const uint2* adj;         // (col, weight bits); hubs' slices are contiguous
    int32_t n;
    const int32_t* srcs;      // [nq] or null (one query from src0)
    int32_t src0;
    void* work;               // DistT[nq * n]
    uint32_t* dist_out;       // [nq * n], or null when work holds the caller's distances
    int32_t* pred_out;        // [nq * n] (PRED != 0)
    uint32_t delta;           // threshold step (u32, or f32 bits)
    uint32_t front;           // vertices waiting in near below which T grows
    // Vertex v waits at place p = v * hash mod 2^bits: bit p mod 2^log_b of
    // word p / 2^log_b.  The hash spreads neighbouring vertices, and so every
    // front, over the words and their owners.
    uint32_t mask;            // 2^bits - 1
    int32_t log_b;            // log2 of the bits used per word (0..5)
    int32_t log_g;            // log2 of the cluster's blocks: word w lives in block w % G
    int32_t words;            // words per block (wave), or in all (tide)
    int32_t hops;             // hops of a warp per step
    int32_t pull;             // breadth-first on a symmetric graph: wide levels are pulled
    int32_t unit;             // breadth-first: every arc weighs 1, hub slices belong to the step that lists them
    int32_t hub_deg;          // a vertex with more arcs is not left to one warp
    int32_t has_hubs;
    uint32_t wide;            // wave: give up (kErrWide) when more vertices than this wait in near
    Ctrl* ctrl;               // error word, finished queries, statistics
    unsigned long long timeout_ns;
    // tide only
    const int32_t* mid;       // [n] end of a row's light arcs (core search), or null
    const uint4* quads;       // [n][2] the first four arcs of every vertex (kNoArc: none; bit 31 of the first: more), or null
    uint32_t light_w;         // weights of light arcs: at most this
    int32_t core_deg;         // a vertex with as many arcs belongs to the core
    int64_t arcs;             // of the graph
    uint32_t* bits;           // near[2], far[2]: `words` words each
    uint4* items;             // hub slices, two lists of items_cap: (vertex, distance, first arc, end)
    uint32_t items_cap;
    struct TideSync* sync;
};

constexpr uint32_t kWaveOwn = 64;      // improved vertices that a warp keeps for its own next hop

constexpr uint32_t kNoArc = 0x7fffffffu;
constexpr int kHopsQuads = 2;          // several hops a step, on graphs with quads

template <int HOPS>
struct WaveLists {
    uint32_t list[64];                 // vertices taken from the words (bit 31: from far)
    uint2 own[2][HOPS ? kWaveOwn : 1]; // (vertex, distance) of this hop and the next
};

struct WaveSlot {
    uint32_t near, fmin, stop, pad;
};

struct WaveHub {
    uint32_t v, d;
    int2 arcs;
};

struct WaveShared {
    WaveSlot slot[2][kWaveMaxCluster];  // what every block of the cluster reports at the end of a step
    uint32_t near[4], fmin[4], nhub[4]; // this block's sums of step s, set s % 4
    WaveHub hub[kWaveHubs];
};

// Grid barriers and the sums of a step (set s % 4).  A block arrives by one
// addition that carries its near count: arrivals in the low 16 bits.
struct __align__(128) TideSync {
    struct __align__(128) {
        unsigned long long arrived;      // end of the step: near count << 16 | blocks
        uint32_t far;                    // the complement of the smallest far distance
        uint32_t core;                   // the complement of the smallest distance that left heavy arcs out
        uint32_t pad[28];
    } set[4];
    struct __align__(128) {
        unsigned long long arcs;         // left out by the core
        unsigned long long pad[15];
    } left;
    struct __align__(128) {
        uint32_t count;                  // hub slices listed by the step
        uint32_t arrived;                // blocks that have listed theirs (breadth-first)
        uint32_t pad[30];
    } hub[4];
};

__device__ __forceinline__ uint32_t cluster_rank() {
    uint32_t r;
    asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
__device__ __forceinline__ void cluster_barrier() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ uint32_t map_rank(uint32_t smem, uint32_t rank) {
    uint32_t a;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(smem), "r"(rank));
    return a;
}
__device__ __forceinline__ void st_cluster(uint32_t a, uint32_t v) {
    asm volatile("st.relaxed.cluster.shared::cluster.u32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}

// Stores of a batch, predicated by hand where most of them happen (thin fronts:
// a branch around each costs more than the store) or behind a branch where
// few arcs improve anything (R-MAT-22 loses 6% without it).
template <bool PREDICATED, typename V>
__device__ __forceinline__ void red_min_if(bool on, V* p, V v) {
    if constexpr (!PREDICATED) {
        if (on) red_min(p, v);
    } else if constexpr (sizeof(V) == 4) {
        asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %2, 0;\n\t@p red.relaxed.gpu.global.min.u32 [%0], %1;\n\t}"
                     ::"l"(p), "r"(v), "r"((uint32_t)on) : "memory");
    } else {
        asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %2, 0;\n\t@p red.relaxed.gpu.global.min.u64 [%0], %1;\n\t}"
                     ::"l"(p), "l"(v), "r"((uint32_t)on) : "memory");
    }
}
__device__ __forceinline__ void st_shared_if(bool on, uint32_t a, uint32_t x, uint32_t y) {
    asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %3, 0;\n\t@p st.shared.v2.u32 [%0], {%1, %2};\n\t}"
                 ::"r"(a), "r"(x), "r"(y), "r"((uint32_t)on) : "memory");
}

// T raised above `base` by delta, and at least above `low` (an f32 delta may
// be absorbed, a u32 sum saturates)
template <int WT>
__device__ __forceinline__ uint32_t wave_raise(uint32_t base, uint32_t delta, uint32_t low) {
    uint32_t t;
    if (WT == 0) {
        t = base + delta;
        if (t < base) t = kInfU32;
    } else {
        t = __float_as_uint(__uint_as_float(base) + __uint_as_float(delta));
        if (t < base) t = base;
    }
    return t > low ? t : low + 1u;
}

// Where the pending bits live: one block's shared memory, a cluster's, or
// global memory.
enum WaveMode { kWaveBlock = 0, kWaveCluster = 1, kWaveGrid = 2 };

// HOPS: a warp may have more than one hop a step (compiled out otherwise: with
// it R-MAT-22 took 8% and R-MAT-13 12% longer at one hop).
// CORE: rows may be relaxed without their heavy arcs (see tide_kernel).
template <int WT, int PRED, int MODE, int HOPS, bool CORE = false>
struct Wave {
    using DistT = typename std::conditional<PRED == 0, uint32_t, unsigned long long>::type;
    using A = Arith<WT>;
    using Addr = typename std::conditional<MODE == kWaveGrid, uint32_t*, uint32_t>::type;

    const WaveParams& P;
    DistT* dist;
    WaveLists<HOPS>* lists;    // this warp's
    uint32_t T, Told;
    Addr near_w, far_w;        // the words written in this step
    uint32_t n_imp, fmin;      // this thread's near improvements and smallest far distance of the step
    uint32_t n_relax;          // arcs relaxed by this thread
    uint32_t n_own, own_w;     // entries kept for the next hop, and which half they are in
    bool keep;                 // the warp has another hop in this step
    uint32_t delta;            // of P, or infinite after the pull
    // CORE: the smallest distance that left heavy arcs out, so far and in this
    // step, the arcs that this thread left out in this step, and the bound from
    // which on distances are of no use
    uint32_t core, left, left_arcs, bound;
    bool skip;                 // CORE: heavy arcs of the core are left out

    static __device__ __forceinline__ uint32_t dpart(uint32_t w) { return w; }
    static __device__ __forceinline__ uint32_t dpart(unsigned long long w) { return (uint32_t)(w >> 32); }

    __device__ __forceinline__ Addr bit_addr(Addr base, uint32_t v, uint32_t& mask) const {
        const uint32_t p = (v * kWaveHash) & P.mask, w = p >> P.log_b;
        mask = 1u << (p & ((1u << P.log_b) - 1u));
        if constexpr (MODE == kWaveGrid) return base + w;
        else if constexpr (MODE == kWaveCluster)
            return map_rank(base + (w >> P.log_g) * 4u, w & ((1u << P.log_g) - 1u));
        else return base + w * 4u;
    }
    // the vertex of bit b of word w
    __device__ __forceinline__ uint32_t vertex(uint32_t w, uint32_t b) const {
        return (((w << P.log_b) | b) * kWaveHashInv) & P.mask;
    }
    __device__ __forceinline__ void red_or(Addr a, uint32_t v) const {
        if constexpr (MODE == kWaveGrid)
            red_or_global(a, v);
        else if constexpr (MODE == kWaveCluster)
            asm volatile("red.relaxed.cluster.shared::cluster.or.b32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
        else asm volatile("red.relaxed.cta.shared::cta.or.b32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
    }

    __device__ __forceinline__ void red_or_if(bool on, Addr a, uint32_t v) const {
        if constexpr (MODE == kWaveGrid)
            asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %2, 0;\n\t@p red.relaxed.gpu.global.or.b32 [%0], %1;\n\t}"
                         ::"l"(a), "r"(v), "r"((uint32_t)on) : "memory");
        else if constexpr (MODE == kWaveCluster)
            asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %2, 0;\n\t"
                         "@p red.relaxed.cluster.shared::cluster.or.b32 [%0], %1;\n\t}"
                         ::"r"(a), "r"(v), "r"((uint32_t)on) : "memory");
        else
            asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %2, 0;\n\t"
                         "@p red.relaxed.cta.shared::cta.or.b32 [%0], %1;\n\t}"
                         ::"r"(a), "r"(v), "r"((uint32_t)on) : "memory");
    }

    // Relaxes K arcs (u at distance du) -> a.x of weight a.y whose distance
    // words are c: lowers dist[v] without waiting for the answer and marks v
    // when the distance beat the loaded one (whoever lowers dist[v] saw a
    // larger value, so the last improvement always marks it).  Straight-line
    // code with predicated stores: as branches, four arcs took 2200 cycles of
    // a 9300-cycle step (grid 256^2 on GB300), like this 300.
    template <int K, bool OWN>
    __device__ __forceinline__ void relax(const uint32_t (&u)[K], const uint32_t (&du)[K], const uint2 (&a)[K],
                                          const DistT (&c)[K], const bool (&in)[K]) {
        uint32_t nd[K], mask[K];
        Addr ad[K];
        bool upd[K], imp[K];
#pragma unroll
        for (int k = 0; k < K; k++) {
            nd[k] = A::add(du[k], P.unit ? 1u : a[k].y);
            const bool use = in[k] && (!CORE || nd[k] < bound);
            if (PRED == 0) {
                upd[k] = imp[k] = use && nd[k] < (uint32_t)c[k];
            } else {
                imp[k] = use && nd[k] < dpart(c[k]);
                upd[k] = PRED == 2 ? imp[k]
                                   : use && (((unsigned long long)nd[k] << 32) | u[k]) < (unsigned long long)c[k];
            }
            ad[k] = bit_addr(nd[k] < T ? near_w : far_w, a[k].x, mask[k]);
        }
#pragma unroll
        for (int k = 0; k < K; k++) {
            if (PRED == 0) {
                red_min_if<HOPS != 0>(upd[k], reinterpret_cast<uint32_t*>(dist) + a[k].x, nd[k]);
            } else {
                unsigned long long* p = reinterpret_cast<unsigned long long*>(dist) + a[k].x;
                const unsigned long long cand = ((unsigned long long)nd[k] << 32) | u[k];
                if (PRED == 1) {
                    red_min_if<HOPS != 0>(upd[k], p, cand);
                } else {
                    unsigned long long x = (unsigned long long)c[k];
                    while (imp[k]) {
                        const unsigned long long old = atomicCAS(p, x, cand);
                        if (old == x) break;
                        x = old;
                        imp[k] = nd[k] < (uint32_t)(x >> 32);
                    }
                }
            }
        }
        if constexpr (!(OWN && HOPS != 0)) {
#pragma unroll
            for (int k = 0; k < K; k++) {
                const bool near = imp[k] && nd[k] < T;
                fmin = imp[k] && !near ? min(fmin, nd[k]) : fmin;
                if (imp[k]) red_or(ad[k], mask[k]);
                n_imp += near ? 1u : 0u;
            }
            return;
        }
        bool near[K], mark[K];
        uint32_t b[K];
#pragma unroll
        for (int k = 0; k < K; k++) {
            near[k] = imp[k] && nd[k] < T;
            mark[k] = imp[k];
            fmin = imp[k] && !near[k] ? min(fmin, nd[k]) : fmin;
            b[k] = __ballot_sync(kFull, near[k]);
        }
        if (keep) {
            // what the warp keeps for its next hop is not marked
            const uint32_t list = (uint32_t)__cvta_generic_to_shared(lists->own[own_w]), lt = lanemask_lt();
            uint32_t at[K], room[K];
#pragma unroll
            for (int k = 0; k < K; k++) {
                at[k] = __popc(b[k] & lt);
                room[k] = __popc(b[k]);
            }
#pragma unroll
            for (int k = 0; k < K; k++) {
                at[k] += n_own;
                n_own += room[k];
                const bool kept = near[k] && at[k] < kWaveOwn;
                st_shared_if(kept, list + at[k] * 8u, a[k].x, nd[k]);
                near[k] = near[k] && !kept;
                mark[k] = mark[k] && !kept;
            }
            n_own = min(n_own, kWaveOwn);
        }
#pragma unroll
        for (int k = 0; k < K; k++) {
            red_or_if(mark[k], ad[k], mask[k]);
            n_imp += near[k] ? 1u : 0u;
        }
    }

    // Up to four arcs of one vertex, `stride` apart, all loads in flight together.
    // (Arc numbers end at 2^31 - 1: those past a row's end are formed unsigned.)
    template <bool OWN>
    __device__ __forceinline__ void arcs4(uint32_t u, uint32_t du, uint32_t e, uint32_t stride, uint32_t end) {
        uint2 a[4];
        DistT c[4];
        uint32_t uu[4], dd[4];
        bool in[4];
#pragma unroll
        for (int k = 0; k < 4; k++) {
            in[k] = e + k * stride < end;
            uu[k] = u;
            dd[k] = du;
            a[k] = in[k] ? ld_arc(P.adj + e + k * stride) : make_uint2(0u, 0u);
        }
#pragma unroll
        for (int k = 0; k < 4; k++) c[k] = in[k] ? ld_dist(dist + a[k].x) : (DistT)0;
        relax<4, OWN>(uu, dd, a, c, in);
    }

    // Arcs g0 + lane + 32 k (k < K) of the warp's concatenated rows (ex: arcs
    // before this lane's vertex u, row at rs, distance du).
    template <int K>
    __device__ __forceinline__ void arcs_packed(uint32_t g0, uint32_t total, uint32_t ex, uint32_t rs, uint32_t du,
                                                uint32_t u) {
        uint2 a[K];
        DistT c[K];
        uint32_t dj[K], uj[K];
        bool in[K];
#pragma unroll
        for (int k = 0; k < K; k++) {
            const uint32_t g = g0 + 32u * k + lane_id();
            int j = 0;
#pragma unroll
            for (int s = 16; s >= 1; s >>= 1)
                if (__shfl_sync(kFull, ex, j + s) <= g) j += s;
            const uint32_t row = __shfl_sync(kFull, rs, j) + (g - __shfl_sync(kFull, ex, j));
            dj[k] = __shfl_sync(kFull, du, j);
            uj[k] = PRED != 0 ? __shfl_sync(kFull, u, j) : 0u;
            in[k] = g < total;
            a[k] = in[k] ? ld_arc(P.adj + row) : make_uint2(0u, 0u);
        }
#pragma unroll
        for (int k = 0; k < K; k++) c[k] = in[k] ? ld_dist(dist + a[k].x) : (DistT)0;
        relax<K, true>(uj, dj, a, c, in);
    }

    // Whether vertex v, of the last hop at distance d or from the words (d
    // infinite), is still to be relaxed, and d: its distance `now`.
    __device__ __forceinline__ bool claim(uint32_t v, bool is_far, uint32_t now, uint32_t& d, bool marks = true) {
        // improved meanwhile: whoever did marked it again
        if (d != kInfU32) return now >= d;
        d = now;
        if (!is_far) return true;
        // below the old threshold: it went through near since
        if (d < Told) return false;
        if (d < T) return true;
        uint32_t mask;
        const Addr a = bit_addr(far_w, v, mask);
        if (marks) red_or(a, mask);
        fmin = min(fmin, d);
        return false;
    }

    // A batch of up to eight vertices, an arc a lane (lanes 4 j to 4 j + 3 have
    // vertex j): on a thin front a batch has three on average, and the chain of
    // instructions from the answers to the next hop is a third as long.
    __device__ __forceinline__ void relax_narrow(bool have, uint32_t v, bool is_far, uint32_t d) {
        const uint32_t k = lane_id() & 3u;
        uint2 a[1] = {make_uint2(kNoArc, 0u)};
        uint32_t now = kInfU32;
        if (have) {
            a[0] = ld_arc(reinterpret_cast<const uint2*>(P.quads) + 4 * (size_t)v + k);
            now = dpart(ld_dist(dist + v));
        }
        const bool more = k == 0u && (a[0].x >> 31) != 0u;
        a[0].x &= kNoArc;
        bool in[1] = {a[0].x != kNoArc};
        const DistT c[1] = {in[0] ? ld_dist(dist + a[0].x) : (DistT)0};
        if (have) have = claim(v, is_far, now, d, k == 0u);
        in[0] = in[0] && have;
        n_relax += in[0] ? 1u : 0u;
        const uint32_t uu[1] = {v}, dd[1] = {d};
        relax<1, true>(uu, dd, a, c, in);
        rest_of(v, d, have && more);
    }
    // The arcs after the fourth of the vertices of lanes `more`.
    __device__ __forceinline__ void rest_of(uint32_t v, uint32_t d, bool more) {
        if (__any_sync(kFull, more)) {
            const int2 sp = more ? __ldg(P.span + v) : make_int2(0, 0);
            const uint32_t end = (uint32_t)sp.y;
            uint32_t e = min((uint32_t)sp.x + 4u, end);
            n_relax += end - e;
            for (; __any_sync(kFull, e < end); e += 4u) arcs4<true>(v, d, e, 1u, end);
        }
        __syncwarp();
    }

    // A batch of relax_batch whose first four arcs lie at a fixed place: two
    // dependent loads (arcs, their ends' distances) instead of three.  The
    // check of the vertex itself comes back meanwhile.  GB300, us: grid 256^2 864
    // -> 768, grid 1024^2 4006 -> 3600, 13 queries on grid 301 x 257 1122 -> 1000;
    // road 4096^2 6006, 5987.
    __device__ __forceinline__ void relax_quads(bool have, uint32_t v, bool is_far, uint32_t d) {
        uint4 x = make_uint4(kNoArc, 0u, kNoArc, 0u), y = x;
        uint32_t now = kInfU32;
        if (have) {
            x = __ldg(P.quads + 2 * (size_t)v);
            y = __ldg(P.quads + 2 * (size_t)v + 1);
            now = dpart(ld_dist(dist + v));
        }
        const bool more = (x.x >> 31) != 0u;
        const uint2 a[4] = {make_uint2(x.x & kNoArc, x.y), make_uint2(x.z, x.w), make_uint2(y.x, y.y), make_uint2(y.z, y.w)};
        DistT c[4];
        bool in[4];
#pragma unroll
        for (int k = 0; k < 4; k++) {
            in[k] = a[k].x != kNoArc;
            c[k] = in[k] ? ld_dist(dist + a[k].x) : (DistT)0;
        }
        if (have) have = claim(v, is_far, now, d);
        const uint32_t uu[4] = {v, v, v, v}, dd[4] = {d, d, d, d};
#pragma unroll
        for (int k = 0; k < 4; k++) {
            in[k] = in[k] && have;
            n_relax += in[k] ? 1u : 0u;
        }
        relax<4, true>(uu, dd, a, c, in);
        rest_of(v, d, have && more);
    }

    // Relaxes up to 32 vertices, one per lane (`have`): from the words
    // (is_far: from the far ones) or, with their distance d, from the warp's
    // last hop.  `hub(v, d, arcs, deg)` takes those with more than hub_deg arcs
    // (it returns the arcs that are left to the warp).
    template <typename Hub>
    __device__ __forceinline__ void relax_batch(bool have, uint32_t v, bool is_far, uint32_t d, bool narrow, Hub&& hub) {
        const uint32_t lane = lane_id();
        if constexpr (HOPS == kHopsQuads) {
            if (narrow) relax_narrow(have, v, is_far, d);
            else relax_quads(have, v, is_far, d);
            return;
        }
        int2 sp = make_int2(0, 0);
        if (have) {
            const uint32_t now = dpart(ld_dist(dist + v));
            sp = P.span ? __ldg(P.span + v) : make_int2(__ldg(P.row + v), __ldg(P.row + v + 1));
            have = claim(v, is_far, now, d);
        }
        if (CORE && skip && have && (sp.y - sp.x >= P.core_deg || d >= core)) {
            const int32_t m = __ldg(P.mid + v);
            if (m < sp.y) left = min(left, d);
            left_arcs += (uint32_t)(sp.y - m);
            sp.y = m;
        }
        int32_t deg = have ? sp.y - sp.x : 0;
        n_relax += (uint32_t)deg;
        if (P.has_hubs) deg = hub(v, d, sp, deg);
        if (__reduce_max_sync(kFull, (uint32_t)deg) <= 4u) {
            // few arcs a vertex: each lane its own
            arcs4<true>(v, d, (uint32_t)sp.x, 1u, (uint32_t)(sp.x + deg));
        } else {
            // the batch's arcs spread over the lanes, 128 at a time
            uint32_t incl = (uint32_t)deg;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t x = __shfl_up_sync(kFull, incl, o);
                if (lane >= (uint32_t)o) incl += x;
            }
            const uint32_t ex = incl - (uint32_t)deg, total = __shfl_sync(kFull, incl, 31);
            if (!P.has_hubs && total <= 32u) arcs_packed<1>(0u, total, ex, (uint32_t)sp.x, d, v);
            else for (uint32_t g0 = 0u; g0 < total; g0 += 128u) arcs_packed<4>(g0, total, ex, (uint32_t)sp.x, d, v);
        }
        __syncwarp();
    }

    // The warp's part of a step.  Hop 0: empties the words i = first,
    // first + stride, ... below `words` (32 at a time: this lane's is i + lane)
    // into the list and relaxes the list's vertices 32 at a time; `take(i, nb,
    // fb)` reads and clears a lane's word.  Then P.hops - 1 hops over the near
    // vertices that the warp itself improved: a hop without the barrier and the
    // words costs half, and a vertex relaxed too early only costs its arcs.
    template <typename Take, typename Vertex, typename Hub>
    __device__ __forceinline__ void sweep(uint32_t first, uint32_t stride, uint32_t words, Take&& take,
                                          Vertex&& vertex_of, Hub&& hub) {
        const uint32_t lane = lane_id();
        uint32_t held = 0u, nb = 0u, fb = 0u, base = first, own = 0u, pos = 0u;
        int32_t hop = 0;
        bool more = base < words;
        n_own = own_w = 0u;
        keep = HOPS && P.hops > 1;
        if (more) take(base + lane, nb, fb);
        for (;;) {
            uint32_t v = 0u, d = kInfU32;
            bool have = false, is_far = false, narrow = false;
            while (more && held < 32u) {
                const bool got = (nb | fb) != 0u;
                const uint32_t m = __ballot_sync(kFull, got);
                if (!m) {
                    base += stride;
                    more = base < words;
                    if (more) take(base + lane, nb, fb);
                    continue;
                }
                if (got) {
                    const uint32_t b = (uint32_t)__ffs((int)(nb | fb)) - 1u;
                    lists->list[held + __popc(m & lanemask_lt())] =
                        vertex_of(base + lane, b) | ((nb >> b) & 1u ? 0u : 0x80000000u);
                    nb &= ~(1u << b);
                    fb &= ~(1u << b);
                }
                held += __popc(m);
                __syncwarp();
            }
            if (held) {
                const uint32_t k = held < 32u ? held : 32u;
                held -= k;
                narrow = HOPS == kHopsQuads && k <= 8u;
                const uint32_t j = narrow ? lane >> 2 : lane;
                have = j < k;
                if (have) v = lists->list[held + j];
                is_far = (v >> 31) != 0u;
                v &= 0x7fffffffu;
            } else if (HOPS && pos < own) {
                narrow = HOPS == kHopsQuads && own - pos <= 8u;
                const uint32_t j = pos + (narrow ? lane >> 2 : lane);
                have = j < own;
                if (have) {
                    const uint2 e = lists->own[own_w ^ 1u][j];
                    v = e.x;
                    d = e.y;
                }
                pos += 32u;
            } else {
                if (!HOPS || n_own == 0u) break;
                hop++;
                keep = hop + 1 < P.hops;
                own = n_own;
                pos = n_own = 0u;
                own_w ^= 1u;
                __syncwarp();
                continue;
            }
            relax_batch(have, v, is_far, d, narrow, hub);
        }
    }

    // The results of vertices first, first + stride, ... (packed words only).
    __device__ __forceinline__ void unpack(size_t out, uint32_t first, uint32_t stride) const {
        if (PRED == 0) return;
        for (uint32_t v = first; v < (uint32_t)P.n; v += stride) {
            const unsigned long long x = __ldcg(reinterpret_cast<const unsigned long long*>(dist) + v);
            uint32_t dd = (uint32_t)(x >> 32);
            if (WT == 1 && dd == kInfU32) dd = kInfF32;
            P.dist_out[out + v] = dd;
            P.pred_out[out + v] = (int32_t)(uint32_t)x;
        }
    }

    __device__ __forceinline__ void init(uint32_t src, uint32_t first, uint32_t stride) const {
        const DistT inf = PRED != 0 ? (DistT)~0ull : (DistT)(WT == 1 ? kInfF32 : kInfU32);
        for (uint32_t v = first; v < (uint32_t)P.n; v += stride)
            dist[v] = v == src ? (DistT)(PRED != 0 ? src : 0u) : inf;
    }

    // The next step's threshold from this step's sums.  Returns 0: no more
    // work, 1: near only, 2: near and the far bits below the new T.
    __device__ __forceinline__ int advance(uint32_t near, uint32_t far_low) {
        if (near < P.front && far_low != kInfU32) {
            Told = T;
            T = near ? wave_raise<WT>(T, delta, 0u) : wave_raise<WT>(max(T, far_low), delta, far_low);
            return 2;
        }
        return near ? 1 : 0;
    }

    // The same while heavy arcs are left out: the threshold stops at `settled`,
    // below which distances are final.  3: they are, and the others are to be
    // pulled.
    __device__ __forceinline__ int advance_core(uint32_t near, uint32_t far_low, uint32_t settled) {
        if (core == kInfU32) return advance(near, far_low);
        if (T >= settled) return near ? 1 : 3;
        const int what = advance(near, far_low);
        T = min(T, settled);
        return what ? what : 3;
    }

    // Vertex v (distance word cur, arcs sp; deg arcs to look at, all of them
    // or none) takes the best of its in-neighbours, its own arcs' ends, of
    // those nearer than `limit`.  The whole warp is here.  Returns its distance
    // after that.
    __device__ __forceinline__ uint32_t pull(uint32_t v, DistT cur, int2 sp, int32_t deg, uint32_t limit) {
        constexpr uint32_t none = PRED == 0 && WT == 1 ? kInfF32 : kInfU32;
        const uint32_t lane = lane_id();
        uint32_t best = none, from = kInfU32;
        auto offer = [&](uint2 a, DistT c) {
            const uint32_t du = dpart(c);
            if (du >= limit) return;
            const uint32_t nd = A::add(du, P.unit ? 1u : a.y);
            if (nd < best || (nd == best && a.x < from)) {
                best = nd;
                from = a.x;
            }
        };
        // (longer rows by the whole warp: R-MAT-22 us at 64, 32, 16, 8 622, 607, 576,
        // 598; R-MAT-20 274, 262, 255, 262)
        const bool by_warp = deg > 16;
        // (of a level, any parent gives the distance)
        for (int32_t e = 0; !by_warp && e < deg && !(PRED == 0 && P.unit && best != none); e += 4) {
            uint2 a[4];
            DistT c[4];
#pragma unroll
            for (int k = 0; k < 4; k++) a[k] = ld_arc(P.adj + sp.x + min(e + k, deg - 1));
#pragma unroll
            for (int k = 0; k < 4; k++) c[k] = ld_dist(dist + a[k].x);
#pragma unroll
            for (int k = 0; k < 4; k++) offer(a[k], c[k]);
        }
        uint32_t m = __ballot_sync(kFull, by_warp);
        while (m) {
            const int j = __ffs((int)m) - 1;
            m &= m - 1u;
            const uint32_t keep_b = best, keep_f = from;
            const uint32_t b = (uint32_t)__shfl_sync(kFull, sp.x, j), end = b + (uint32_t)__shfl_sync(kFull, deg, j);
            best = none;
            from = kInfU32;
            for (uint32_t e = b; e < end; e += 128u) {
                uint2 a[4];
                DistT c[4];
#pragma unroll
                for (int k = 0; k < 4; k++) a[k] = ld_arc(P.adj + min(e + 32u * k + lane, end - 1u));
#pragma unroll
                for (int k = 0; k < 4; k++) c[k] = ld_dist(dist + a[k].x);
#pragma unroll
                for (int k = 0; k < 4; k++) offer(a[k], c[k]);
            }
            const uint32_t mb = __reduce_min_sync(kFull, best);
            const uint32_t mf = __reduce_min_sync(kFull, best == mb ? from : kInfU32);
            best = (int)lane == j ? mb : keep_b;
            from = (int)lane == j ? mf : keep_f;
        }
        const uint32_t d = dpart(cur);
        if (deg > 0 && best != none) {
            if (PRED == 0) {
                if (best < d) reinterpret_cast<volatile uint32_t*>(dist)[v] = best;
            } else {
                const unsigned long long cand = ((unsigned long long)best << 32) | from;
                if (PRED == 1 ? cand < (unsigned long long)cur : best < d)
                    reinterpret_cast<volatile unsigned long long*>(dist)[v] = cand;
            }
        }
        return deg > 0 ? min(d, best) : d;
    }

    __device__ __forceinline__ void publish(uint32_t improved) const {
        unsigned long long r64 = n_relax, i64 = improved;
        for (int o = 16; o > 0; o >>= 1) {
            r64 += __shfl_down_sync(kFull, r64, o);
            i64 += __shfl_down_sync(kFull, i64, o);
        }
        if (lane_id() == 0 && r64) {
            atomicAdd(&P.ctrl->stats[kStRelax], r64);
            atomicAdd(&P.ctrl->stats[kStImproved], i64);
        }
    }
};

// One cluster (CL) or one block per query.  The blocks exchange a step's sums
// by writing them into every block's slots; one cluster barrier then makes
// them and the step's marks visible.  Two slot sets alternate: a block can
// write set s + 2 only after all blocks passed barrier s + 1, after reading s.
template <int WT, int PRED, bool CL, int HOPS>
__global__ void __launch_bounds__(1024, 1) wave_kernel(const __grid_constant__ WaveParams P) {
    using W = Wave<WT, PRED, CL ? kWaveCluster : kWaveBlock, HOPS>;
    using DistT = typename W::DistT;
    extern __shared__ __align__(16) uint32_t wave_words[];   // near[2], far[2]
    __shared__ WaveShared S;
    __shared__ WaveLists<HOPS> lists[32];
    const uint32_t tid = threadIdx.x, nt = blockDim.x, lane = tid & 31u;
    const uint32_t G = CL ? 1u << P.log_g : 1u, rank = CL ? cluster_rank() : 0u;
    const uint32_t q = CL ? blockIdx.x >> P.log_g : blockIdx.x;
    const uint32_t src = (uint32_t)(P.srcs ? P.srcs[q] : P.src0);
    const uint32_t words = (uint32_t)P.words;
    W w{P, reinterpret_cast<DistT*>(P.work) + (size_t)q * (size_t)P.n, &lists[tid >> 5],
        wave_raise<WT>(0u, P.delta, 0u), 0u, 0u, 0u, 0u, kInfU32, 0u, 0u, 0u, false, P.delta, kInfU32, kInfU32, 0u, kInfU32, false};

    // every distance to infinity but the source's, and its pending bit
    w.init(src, rank * nt + tid, G * nt);
    for (uint32_t i = tid; i < 4u * words; i += nt) wave_words[i] = 0u;
    if (tid < 4u) {
        S.near[tid] = S.nhub[tid] = 0u;
        S.fmin[tid] = kInfU32;
    }
    __syncthreads();
    {
        const uint32_t p = (src * kWaveHash) & P.mask, sw = p >> P.log_b;
        if (tid == 0 && (sw & (G - 1u)) == rank) wave_words[sw >> P.log_g] = 1u << (p & ((1u << P.log_b) - 1u));
    }
    if (CL) cluster_barrier();
    else __syncthreads();

    uint32_t cur = 0u, fw = 0u, far_low = kInfU32;   // far_low: no far vertex lies below it
    uint32_t n_improved = 0, steps = 0;
    const unsigned long long deadline = gtime() + P.timeout_ns;
    int error = kErrNone, what = 1;
    while (what) {
        const uint32_t par = steps & 1u, set = steps & 3u;
        const bool scan_far = what == 2;
        uint32_t* near_r = wave_words + cur * words;
        uint32_t* far_r = wave_words + (2u + fw) * words;
        if (scan_far) fw ^= 1u;
        cur ^= 1u;
        w.near_w = (uint32_t)__cvta_generic_to_shared(wave_words + cur * words);
        w.far_w = (uint32_t)__cvta_generic_to_shared(wave_words + (2u + fw) * words);
        w.n_imp = 0u;
        w.fmin = kInfU32;
        w.sweep(
            tid & ~31u, nt, words,
            [&](uint32_t i, uint32_t& nb, uint32_t& fb) {
                nb = fb = 0u;
                if (i < words) {
                    nb = near_r[i];
                    if (nb) near_r[i] = 0u;
                    if (scan_far) {
                        fb = far_r[i];
                        if (fb) far_r[i] = 0u;
                        fb &= ~nb;
                    }
                }
            },
            [&](uint32_t i, uint32_t b) { return w.vertex((i << P.log_g) | rank, b); },
            [&](uint32_t v, uint32_t d, int2 sp, int32_t deg) {
                if (deg <= P.hub_deg) return deg;
                const uint32_t h = atomicAdd(&S.nhub[set], 1u);
                if (h >= (uint32_t)kWaveHubs) return deg;
                S.hub[h] = WaveHub{v, d, sp};
                return 0;
            });
        if (P.has_hubs) {
            // a hub is expanded by its whole block
            __syncthreads();
            const uint32_t nh = min(S.nhub[set], (uint32_t)kWaveHubs);
            for (uint32_t h = 0; h < nh; h++) {
                const WaveHub hb = S.hub[h];
                const uint32_t end = (uint32_t)hb.arcs.y;
                for (uint32_t e = (uint32_t)hb.arcs.x + tid; e < end; e += 4u * nt)
                    w.template arcs4<false>(hb.v, hb.d, e, nt, end);
            }
        }
        // the step's sums
        n_improved += w.n_imp;
        const uint32_t imp = __reduce_add_sync(kFull, w.n_imp), fm = __reduce_min_sync(kFull, w.fmin);
        if (lane == 0) {
            if (imp) atomicAdd(&S.near[set], imp);
            if (fm != kInfU32) atomicMin(&S.fmin[set], fm);
        }
        __syncthreads();
        // set s + 2 is empty before anyone adds to it: that comes after the
        // next step's __syncthreads
        if (tid == 0) {
            const uint32_t z = (steps + 2u) & 3u;
            S.near[z] = S.nhub[z] = 0u;
            S.fmin[z] = kInfU32;
        }
        uint32_t near, sfm, stop = 0u;
        if (CL) {
            if (tid < G) {
                const uint32_t a = map_rank((uint32_t)__cvta_generic_to_shared(&S.slot[par][rank]), tid);
                st_cluster(a, S.near[set]);
                st_cluster(a + 4u, S.fmin[set]);
                if (rank == 0) st_cluster(a + 8u, (steps & 255u) == 255u && gtime() > deadline);
            }
            cluster_barrier();
            const bool in = lane < G;
            near = __reduce_add_sync(kFull, in ? S.slot[par][lane].near : 0u);
            sfm = __reduce_min_sync(kFull, in ? S.slot[par][lane].fmin : kInfU32);
            stop = S.slot[par][0].stop;
        } else {
            near = S.near[set];
            sfm = S.fmin[set];
            if ((steps & 255u) == 255u) stop = __syncthreads_or(gtime() > deadline);
        }
        steps++;
        far_low = scan_far ? sfm : min(far_low, sfm);
        what = w.advance(near, far_low);
        if (what && (stop || near > P.wide)) {
            error = stop ? kErrTimeout : kErrWide;
            break;
        }
    }
    w.unpack((size_t)q * (size_t)P.n, rank * nt + tid, G * nt);
    w.publish(n_improved);
    if (rank == 0 && tid == 0) {
        atomicAdd(&P.ctrl->stats[kStIter], (unsigned long long)steps);
        if (error) raise_error(P.ctrl, error, 20, (int)q);
        else atomicAdd(&P.ctrl->finished, 1);
    }
}

// One thread's wait until the word's low 16 bits say that all blocks have
// arrived (launched cooperatively: all are resident); the word, or 0 after
// the deadline.
__device__ __forceinline__ unsigned long long tide_wait(const unsigned long long* p, uint32_t blocks,
                                                        unsigned long long deadline) {
    for (uint32_t spins = 1;; spins++) {
        const unsigned long long x = ld_acquire64(p);
        if ((x & 0xffffull) == blocks) return x;
        if ((spins & 1023u) == 0 && gtime() > deadline) return 0ull;
    }
}
__device__ __forceinline__ void red_release64(unsigned long long* p, unsigned long long v) {
    asm volatile("red.release.gpu.global.add.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

// Breadth-first on a symmetric graph, a level of more vertices than these
// fractions of those not reached yet and of all is pulled: every vertex not
// reached looks for the level in its own row.  On power-law graphs nearly all
// arcs belong to the level before the widest, and lead back.  R-MAT-22 us, with
// parents 783 -> 312, levels only 725 -> 238; R-MAT-20 290 -> 200 (231 at a
// 14th of those not reached; at 1000ths R-MAT-22 pulls too early, 1104), R-MAT-16
// 106 -> 89.
constexpr uint32_t kPullUnreached = 50u, kPullAll = 64u;

// The whole grid on one query.
//
// CORE (symmetric graphs with hubs, light arcs first in every row): most arcs
// belong to hubs that lie close together, and most of those lead to vertices
// that are nearer by other ways.  So vertices of core_deg arcs or more relax
// only their light arcs, and, from the first of them on (at distance `core`),
// all vertices.  What is left out reaches no vertex below core + light_w: up
// to there the search goes on as ever, and what it finds is final.  Then every
// other vertex with arcs looks at all its in-neighbours once (its own arcs,
// reversed), which covers all that was left out, and the search ends among
// these vertices with all their arcs.  On R-MAT-22 from a source of the giant
// component a fifth as many arcs as there are is relaxed or looked at in all.
template <int WT, int PRED, int HOPS, bool CORE>
__global__ void __launch_bounds__(1024, 1) tide_kernel(const __grid_constant__ WaveParams P) {
    using W = Wave<WT, PRED, kWaveGrid, HOPS, CORE>;
    using DistT = typename W::DistT;
    __shared__ WaveLists<HOPS> lists[32];
    __shared__ uint32_t s_near[4], s_fmin[4], s_left[4], s_arcs[4], s_out[4];
    const uint32_t tid = threadIdx.x, nt = blockDim.x, lane = tid & 31u;
    const uint32_t gt = blockIdx.x * nt + tid, gn = gridDim.x * nt;
    // consecutive warps of the grid lie in different blocks
    const uint32_t wid = (tid >> 5) * gridDim.x + blockIdx.x, nw = gn >> 5;
    const uint32_t words = (uint32_t)P.words;
    W w{P, reinterpret_cast<DistT*>(P.work), &lists[tid >> 5],
        wave_raise<WT>(0u, P.delta, 0u), 0u, nullptr, nullptr, 0u, kInfU32, 0u, 0u, 0u, false, P.delta, kInfU32, kInfU32, 0u, kInfU32, false};
    const unsigned long long deadline = gtime() + P.timeout_ns;

    w.init((uint32_t)P.src0, gt, gn);
    for (uint32_t i = gt; i < words; i += gn) {
        const uint32_t p = ((uint32_t)P.src0 * kWaveHash) & P.mask;
        P.bits[i] = i == p >> P.log_b ? 1u << (p & ((1u << P.log_b) - 1u)) : 0u;
        P.bits[words + i] = P.bits[2u * words + i] = P.bits[3u * words + i] = 0u;
    }
    if (tid < 4u) {
        s_near[tid] = 0u;
        s_fmin[tid] = s_left[tid] = kInfU32;
        s_arcs[tid] = 0u;
    }
    w.skip = CORE && !P.unit;

    // step 0 ends the preparation; the searching steps follow
    uint32_t cur = 0u, fw = 0u, far_low = kInfU32, n_improved = 0, steps = 0, near = 0u, settled = kInfU32, reached = 1u;
    int what = 1;
    bool ok = true;
    for (;;) {
        // the step's sums: the block's, then the grid's
        const uint32_t set = steps & 3u;
        const bool scanned = what == 2;
        if (steps) {
            n_improved += w.n_imp;
            const uint32_t imp = __reduce_add_sync(kFull, w.n_imp), fm = __reduce_min_sync(kFull, w.fmin);
            if (lane == 0) {
                if (imp) atomicAdd(&s_near[set], imp);
                if (fm != kInfU32) atomicMin(&s_fmin[set], fm);
            }
            if (CORE && w.skip) {
                const uint32_t left = __reduce_min_sync(kFull, w.left);
                const uint32_t arcs = __reduce_add_sync(kFull, w.left_arcs);
                if (lane == 0 && left != kInfU32) atomicMin(&s_left[set], left);
                if (lane == 0 && arcs) atomicAdd(&s_arcs[set], arcs);
            }
        }
        __syncthreads();
        if (tid == 0) {
            const uint32_t z = (steps + 2u) & 3u;
            if (CORE && s_left[set] != kInfU32) {
                atomicMax(&P.sync->set[set].core, ~s_left[set]);
                atomicAdd(&P.sync->left.arcs, (unsigned long long)s_arcs[set]);
            }
            if (s_fmin[set] != kInfU32) atomicMax(&P.sync->set[set].far, ~s_fmin[set]);
            if (blockIdx.x == 0 && steps) {
                // nobody touches set s + 2 before the barrier after this one
                P.sync->set[z].arrived = 0ull;
                P.sync->set[z].far = P.sync->set[z].core = P.sync->hub[z].count = P.sync->hub[z].arrived = 0u;
            }
            red_release64(&P.sync->set[set].arrived, ((unsigned long long)s_near[set] << 16) | 1ull);
            s_near[z] = 0u;
            s_fmin[z] = s_left[z] = kInfU32;
            s_arcs[z] = 0u;
            const unsigned long long x = tide_wait(&P.sync->set[set].arrived, gridDim.x, deadline);
            s_out[0] = x ? (uint32_t)min(x >> 16, 0xfffffffeull) : kInfU32;
            s_out[1] = ~ld_relaxed(&P.sync->set[set].far);
            s_out[2] = ld_relaxed(&P.sync->hub[set].count);
            if (CORE) s_out[3] = ~ld_relaxed(&P.sync->set[set].core);
        }
        __syncthreads();
        near = s_out[0];
        uint32_t items = P.has_hubs && steps && !P.unit ? s_out[2] : 0u;
        if (near == kInfU32) {
            ok = false;
            break;
        }
        if (steps == 0) {
            near = 1u;
        } else {
            far_low = scanned ? s_out[1] : min(far_low, s_out[1]);
            if (CORE && w.skip) {
                w.core = min(w.core, s_out[3]);
                w.bound = settled = w.core != kInfU32 ? Arith<WT>::add(w.core, P.light_w) : kInfU32;
                what = w.advance_core(near + items, far_low, settled);
            } else {
                what = w.advance(near + items, far_low);
            }
            if (!what) break;
            if (CORE && P.pull) {
                reached = min((uint32_t)P.n, reached + near);
                if (near >= max(((uint32_t)P.n - reached) / kPullUnreached, (uint32_t)P.n / kPullAll)) what = 3;
            }
        }
        const uint32_t prev = set;
        steps++;
        const uint32_t now = steps & 3u;
        if (CORE && what == 3) {
            // nobody waits below `settled`: the others pull, and wait.  Where
            // the core has not settled yet (less than half of the arcs left
            // out) pulling would cost more than relaxing everything again.
            // A wide level: those not reached yet look for a parent in it.
            const bool level = P.unit != 0;
            const bool pulls = level || ld_relaxed64(&P.sync->left.arcs) * 2ull >= (unsigned long long)P.arcs;
            const uint32_t limit = level ? steps : PRED == 0 && WT == 1 ? kInfF32 : kInfU32;
            w.skip = false;
            w.bound = kInfU32;
            if (level) {
                for (uint32_t i = gt; i < words; i += gn) P.bits[(size_t)cur * words + i] = 0u;
                cur ^= 1u;
                settled = PRED == 0 && WT == 1 ? kInfF32 : kInfU32;
            }
            // little is left after the pull: no order among it any more
            if (pulls) w.delta = WT == 1 ? kInfF32 : kInfU32;
            w.near_w = P.bits + (size_t)cur * words;
            w.far_w = P.bits + (size_t)(2u + fw) * words;
            w.n_imp = 0u;
            w.fmin = kInfU32;
            uint32_t v = wid * 32u + lane;
            DistT dv_next = 0;
            int2 sp_next = make_int2(0, 0);
            auto fetch = [&](uint32_t u) {
                if (u < (uint32_t)P.n) {
                    dv_next = ld_dist(w.dist + u);
                    sp_next = __ldg(P.span + u);
                }
            };
            fetch(v);
            for (uint32_t base = wid * 32u; base < (uint32_t)P.n; base += nw * 32u, v += nw * 32u) {
                const bool in = v < (uint32_t)P.n;
                const DistT dv = dv_next;
                const int2 sp = sp_next;
                fetch(v + nw * 32u);
                const int32_t deg = in ? sp.y - sp.x : 0;
                const int32_t look = pulls && W::dpart(dv) >= settled ? deg : 0;
                if (!__any_sync(kFull, pulls ? look > 0 : deg > 0)) continue;
                w.n_relax += (uint32_t)look;
                const uint32_t d = w.pull(v, dv, sp, look, limit);
                // (a vertex with one arc has nobody to tell but its source)
                if ((pulls ? look > 1 : deg > 0) && d != (PRED == 0 && WT == 1 ? kInfF32 : kInfU32)) {
                    uint32_t mask;
                    uint32_t* const a = w.bit_addr(d < w.T ? w.near_w : w.far_w, v, mask);
                    w.red_or(a, mask);
                    if (d < w.T) w.n_imp++;
                    else w.fmin = min(w.fmin, d);
                }
            }
            continue;
        }
        const bool scan_far = what == 2;
        uint32_t* near_r = P.bits + (size_t)cur * words;
        uint32_t* far_r = P.bits + (size_t)(2u + fw) * words;
        if (scan_far) fw ^= 1u;
        cur ^= 1u;
        w.near_w = P.bits + (size_t)cur * words;
        w.far_w = P.bits + (size_t)(2u + fw) * words;
        w.n_imp = 0u;
        w.fmin = w.left = kInfU32;
        w.left_arcs = 0u;
        uint4* items_w = P.items + (size_t)(steps & 1u) * P.items_cap;
        w.sweep(
            wid * 32u, nw * 32u, words,
            [&](uint32_t i, uint32_t& nb, uint32_t& fb) {
                nb = fb = 0u;
                if (i < words) {
                    nb = __ldcg(near_r + i);
                    if (scan_far) fb = __ldcg(far_r + i);
                    if (nb) near_r[i] = 0u;
                    if (fb) far_r[i] = 0u;
                    fb &= ~nb;
                }
            },
            [&](uint32_t i, uint32_t b) { return w.vertex(i, b); },
            [&](uint32_t v, uint32_t d, int2 sp, int32_t deg) {
                // hubs are cut into slices for all warps of the grid
                uint32_t m = __ballot_sync(kFull, deg > P.hub_deg);
                if (deg > P.hub_deg) deg = 0;
                while (m) {
                    const int j = __ffs((int)m) - 1;
                    m &= m - 1u;
                    const uint32_t u = __shfl_sync(kFull, v, j), du = __shfl_sync(kFull, d, j);
                    const uint32_t b = (uint32_t)__shfl_sync(kFull, sp.x, j), e = (uint32_t)__shfl_sync(kFull, sp.y, j);
                    const uint32_t k = (e - b + kTideChunk - 1u) / kTideChunk;
                    uint32_t at = 0;
                    if (lane == 0) at = atomicAdd(&P.sync->hub[now].count, k);
                    at = __shfl_sync(kFull, at, 0);
                    for (uint32_t i = lane; i < k; i += 32u) {
                        const uint32_t lo = b + i * kTideChunk;
                        items_w[at + i] = make_uint4(u, du, lo, min(e, lo + kTideChunk));
                    }
                }
                return deg;
            });
        if (!P.has_hubs) continue;
        const uint4* items_r;
        if (P.unit) {
            // breadth-first: the slices belong to this level
            __syncthreads();
            if (tid == 0) {
                unsigned int x;
                asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(&P.sync->hub[now].arrived) : "memory");
                uint32_t spins = 0;
                ok = true;
                while ((x = ld_acquire(&P.sync->hub[now].arrived)) != gridDim.x)
                    if ((++spins & 1023u) == 0 && gtime() > deadline) {
                        ok = false;
                        break;
                    }
                s_out[2] = ok ? ld_relaxed(&P.sync->hub[now].count) : kInfU32;
            }
            __syncthreads();
            items = s_out[2];
            items_r = items_w;
            if (items == kInfU32) {
                ok = false;
                break;
            }
        } else {
            // the slices that the last step listed, but for those whose hub
            // has improved since: it waits again with its new distance
            items_r = P.items + (size_t)(prev & 1u) * P.items_cap;
        }
        for (uint32_t i = wid; i < items; i += nw) {
            const uint4 it = __ldcg(items_r + i);
            if (!P.unit && W::dpart(ld_dist(w.dist + it.x)) < it.y) continue;
            for (uint32_t e = it.z + lane; e < it.w; e += 128u) w.template arcs4<false>(it.x, it.y, e, 32u, it.w);
            __syncwarp();
        }
    }
    if (ok) w.unpack(0, gt, gn);
    w.publish(n_improved);
    if (tid == 0 && !ok) raise_error(P.ctrl, kErrTimeout, 21, 0);
    if (gt == 0) {
        atomicAdd(&P.ctrl->stats[kStIter], (unsigned long long)steps);
        atomicAdd(&P.ctrl->finished, 1);
    }
}

}  // namespace sssp
