// fan.cuh -- 32 searches of one graph at once, one per lane of a warp.
//
// Searches from many sources over a small-world graph relax the same arcs at
// about the same step.  Run one by one (or through one queue) every arc costs
// a random 4-byte access per query.  Here the distances of a group of 32
// queries lie side by side, one 128-byte row per vertex, and a warp relaxes
// an arc for all of them: one row load, one add and compare per lane, one
// vote, and a reduction by the lanes that improved.  A vertex waits with one
// word whose bits are the queries that improved it.
//
// The grid steps over the waiting vertices in Bellman-Ford order: the queries
// are then aligned by hops.  Ordered by distance a query relaxes an arc 1.2
// times instead of 4, but the queries reach a vertex at different steps, and
// the visits are as many (R-MAT-20, 32 queries, all arcs: 5.4 visits an arc by
// hops, 7 to 8 by distance in simulation).
//
// Per step: list the waiting vertices (long rows in slices, short rows
// whole), grid barrier, relax the lists, grid barrier.
//
// CORE (symmetric graphs with hubs, as in tide_kernel): each query leaves out
// the heavy arcs of the core's vertices, and of all others from the distance
// on where it met the core, and stops at that distance plus the light bound.
// When nobody waits, the vertices beyond pull over their own rows and the
// search ends among them.  In simulation, 32 queries on R-MAT-18: 0.4 visits an
// arc in the core, 0.2 in the pull.
//
// GB300, ms: 256 queries on R-MAT-20 137.7 through the queues, 43.6 here with
// all arcs, 13.8 with the core search; 64 on R-MAT-18 f32 21.1, 5.4, 2.3; 40 on
// R-MAT-17 with predecessors 2.2, 1.4 (all arcs, core); 40 on G(200K, 2M) with
// predecessors 12.8 through the queues, 5.5 here.  With all arcs it is bound by
// instructions and their latency (59% of the issue slots, 39% of the L1
// wavefronts, 14% of L2; 30 G visits of 32 queries a second): 1024 threads of
// 64 registers beat 768 of 80.  The core search is bound by the latency of its
// 18 steps, each of a few items per warp.
#pragma once

#include "wave.cuh"

namespace sssp {

// Rows up to kFanShort arcs are relaxed kFanRows at a time, longer ones in
// slices of kFanChunk.  64 queries on R-MAT-20, us: slices of 128 3630, 64 3430,
// 32 3740; at 128, 8 rows of up to 8 arcs 4230, 16 4060, 32 rows of up to 16 4270.
constexpr int32_t kFanShort = 16;
constexpr uint32_t kFanRows = 8;
constexpr uint32_t kFanChunk = 64;
constexpr int kFanThreads = 1024;
constexpr int32_t kFanCoreArcs = 128; // a vertex with as many arcs belongs to the core
constexpr int32_t kFanMaxVertices = 1 << 25;   // rows are addressed by 32-bit byte offsets

struct FanSync {
    struct __align__(128) {
        uint32_t arrived;
        uint32_t pad[31];
    } barrier;
    struct __align__(128) {
        uint32_t slices, rows;        // listed by the step: slices, short rows
        uint32_t pad0[30];
        uint32_t claimed;             // slices and batches of short rows taken by warps
        uint32_t pad1[31];
    } set[4];
    uint32_t core[32];                // per query: the complement of the smallest distance that left heavy arcs out
};

struct FanParams {
    const int2* span;
    const uint2* adj;
    const int32_t* mid;       // [n] end of a row's light arcs (core search), or null
    uint32_t light_w;         // their largest weight
    int32_t core_deg;         // kFanCoreArcs
    int32_t n;
    int32_t nq;               // queries of this group (1..32)
    const int32_t* srcs;      // [nq]
    uint32_t* dist;           // [n][32]
    uint32_t* pred;           // [n][32] or null: smallest tight in-neighbour, found after the distances
    uint32_t* wait;           // [2][places]: queries that improved the vertex at place v * hash & mask
    uint32_t mask;
    uint4* slices;            // (vertex, queries, first arc, end)
    uint4* rows;              // the same of short rows
    FanSync* sync;
    Ctrl* ctrl;
    unsigned long long timeout_ns;
    // From step max_steps on the search gives up (kErrDeep) where more wait than a
    // tail that the bulk left behind, whose steps cost 12 us (a power-law graph
    // with a chain of 300 arcs: 3.5 ms, 0.9 with 50), or after 16 times as many.
    uint32_t max_steps;
};

constexpr uint32_t kFanTail = 1024;   // slices and short rows of a step

// How an arc is used: to relax it, (distances final) to find the tight ones,
// to relax it while the core leaves heavy arcs out, or to pull over it, from
// its end to the row's vertex.
enum FanPass { kFanRelax = 0, kFanTight = 1, kFanCore = 2, kFanPull = 3 };

template <int WT, int PASS>
struct Fan {
    const FanParams& P;
    uint32_t* wait_w;
    uint32_t lane;
    uint32_t core, bound;     // this lane's query: where heavy arcs are left out from, and up to where that changes nothing

    static constexpr uint32_t kInf = WT == 1 ? kInfF32 : kInfU32;

    __device__ __forceinline__ Fan(const FanParams& p, uint32_t* w) : P(p), wait_w(w), lane(lane_id()) {
        if (PASS == kFanCore || PASS == kFanPull) {
            core = ~__ldcg(P.sync->core + lane);
            bound = core == kInfU32 ? kInf : Arith<WT>::add(core, P.light_w);
        }
    }

    // du (+) w: for whole weights du + min(w, cap) with cap = the largest
    // length - du, which saturates in two instructions (0 from an infinite du)
    static __device__ __forceinline__ uint32_t cap(uint32_t du) { return du == kInfU32 ? 0u : kSatU32 - du; }
    static __device__ __forceinline__ uint32_t add(uint32_t du, uint32_t cap, uint32_t w) {
        return WT == 0 ? du + min(w, cap) : Arith<1>::add(du, w);
    }

    // Byte offset of this lane's distance in the row of a vertex.
    __device__ __forceinline__ uint32_t at(uint32_t v) const { return v * 128u + lane * 4u; }
    __device__ __forceinline__ uint32_t* word(uint32_t* base, uint32_t off) const {
        return reinterpret_cast<uint32_t*>(reinterpret_cast<char*>(base) + off);
    }

    // Eight arcs of which lane j0 + k holds number k, from the distances du(k)
    // (a query that does not take part has an infinite one, which improves
    // nothing): the rows are loaded together.  Adds to `won` of lane j0 + k
    // the queries that arc k improved.  The loop is bound by its instructions,
    // so that the reduction is predicated by hand.
    template <typename From>
    __device__ __forceinline__ void use8(uint2 a, uint32_t u, From&& du, uint32_t j0, uint32_t& won) const {
        uint32_t off[8], cur[8];
#pragma unroll
        for (int k = 0; k < 8; k++) {
            off[k] = at(__shfl_sync(kFull, a.x, j0 + k));
            cur[k] = __ldcg(word(P.dist, off[k]));
        }
#pragma unroll
        for (int k = 0; k < 8; k++) {
            const uint2 d = du(k);
            const uint32_t w = __shfl_sync(kFull, a.y, j0 + k);
            const uint32_t nd = PASS == kFanPull ? add(cur[k], cap(cur[k]), w) : add(d.x, d.y, w);
            if (PASS == kFanPull) off[k] = at(__shfl_sync(kFull, u, j0 + k));
            if (PASS == kFanTight) {
                const uint32_t uk = __shfl_sync(kFull, u, j0 + k);
                if (d.x != kInfU32 && nd == cur[k]) red_min(word(P.pred, off[k]), uk);
            } else {
                uint32_t b;
                asm volatile(
                    "{\n\t.reg .pred p;\n\t"
                    "setp.lt.u32 p, %2, %3;\n\t"
                    "@p red.relaxed.gpu.global.min.u32 [%1], %2;\n\t"
                    "vote.sync.ballot.b32 %0, p, 0xffffffff;\n\t}"
                    : "=r"(b) : "l"(word(P.dist, off[k])), "r"(nd),
                      "r"(PASS == kFanPull ? d.x : PASS == kFanCore ? min(cur[k], bound) : cur[k]) : "memory");
                if (lane == j0 + k) won = b;
            }
        }
    }
    __device__ __forceinline__ void wake(uint32_t v, uint32_t won) const {
        if (PASS != kFanTight && won) red_or_global(wait_w + ((v * kWaveHash) & P.mask), won);
    }

    // A slice of one row: its arcs 32 at a time, one per lane, the next 32 on
    // their way meanwhile.  Lanes past the end hold the last arc again: to
    // relax it twice changes nothing.
    __device__ __forceinline__ void slice(uint4 it) const {
        const uint32_t end = it.w;
        uint2 next = ld_arc(P.adj + min(it.z + lane, end - 1u));
        uint32_t d = __ldcg(word(P.dist, at(it.x)));
        const bool on = (it.y >> lane) & 1u;
        if (PASS == kFanPull) {
            uint32_t best = kInf;
            for (uint32_t e = it.z; e < end; e += 32u) {
                const uint32_t cnt = min(32u, end - e);
                const uint2 a = next;
                next = ld_arc(P.adj + min(e + 32u + lane, end - 1u));
                for (uint32_t j0 = 0; j0 < cnt; j0 += 8u) {
                    uint32_t c[8];
#pragma unroll
                    for (int k = 0; k < 8; k++) c[k] = __ldcg(word(P.dist, at(__shfl_sync(kFull, a.x, j0 + k))));
#pragma unroll
                    for (int k = 0; k < 8; k++)
                        best = min(best, add(c[k], cap(c[k]), __shfl_sync(kFull, a.y, j0 + k)));
                }
            }
            const bool better = on && best < d;
            if (better) red_min(word(P.dist, at(it.x)), best);
            const uint32_t won = __ballot_sync(kFull, better);
            if (lane == 0) wake(it.x, won);
            return;
        }
        if (!on) d = kInf;
        const uint2 from = make_uint2(d, cap(d));
        for (uint32_t e = it.z; e < end; e += 32u) {
            const uint32_t cnt = min(32u, end - e);
            const uint2 a = next;
            next = ld_arc(P.adj + min(e + 32u + lane, end - 1u));
            uint32_t won = 0u;
            for (uint32_t j0 = 0; j0 < cnt; j0 += 8u) use8(a, it.x, [&](int) { return from; }, j0, won);
            wake(a.x, won);
        }
    }

    // Up to 32 short rows, one per lane (v, queries m, deg arcs from begin):
    // their arcs packed 32 at a time, one per lane (past the end the last one).
    __device__ __forceinline__ void rows(uint32_t v, uint32_t m, int32_t begin, int32_t deg) const {
        int32_t incl = deg;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int32_t x = __shfl_up_sync(kFull, incl, o);
            if (lane >= (uint32_t)o) incl += x;
        }
        const int32_t ex = incl - deg, total = __shfl_sync(kFull, incl, 31);
        for (int32_t g0 = 0; g0 < total; g0 += 32) {
            const int32_t g = min(g0 + (int32_t)lane, total - 1);
            int i = 0;
#pragma unroll
            for (int s = 16; s >= 1; s >>= 1)
                if (__shfl_sync(kFull, ex, i + s) <= g) i += s;
            const int32_t arc = __shfl_sync(kFull, begin, i) + (g - __shfl_sync(kFull, ex, i));
            const uint32_t u = __shfl_sync(kFull, v, i), mu = __shfl_sync(kFull, m, i);
            const int32_t row_arcs = PASS == kFanPull ? __shfl_sync(kFull, deg, i) : 0;
            const uint2 a = ld_arc(P.adj + arc);
            const uint32_t cnt = (uint32_t)min(32, total - g0);
            uint32_t won = 0u;
            for (uint32_t j0 = 0; j0 < cnt; j0 += 8u) {
                uint32_t du[8];
#pragma unroll
                for (uint32_t k = 0; k < 8u; k++) {
                    const uint32_t uk = __shfl_sync(kFull, u, j0 + k), mk = __shfl_sync(kFull, mu, j0 + k);
                    du[k] = __ldcg(word(P.dist, at(uk)));
                    if (!((mk >> lane) & 1u)) du[k] = PASS == kFanPull ? 0u : kInf;
                }
                use8(a, u, [&](int k) { return make_uint2(du[k], cap(du[k])); }, j0, won);
            }
            if (PASS != kFanPull) wake(a.x, won);
            else if (row_arcs > 1) wake(u, won);
        }
    }

    // The step's lists: slices, then the short rows kFanRows at a time.  The first
    // seven eighths are dealt out, the rest claimed one by one (one counter
    // gives a claim every nanosecond: with every slice claimed, a step on
    // G(200K, 2M) was bound by it).  While a slice is relaxed, the next one is
    // on its way and the claim after that too.
    __device__ __forceinline__ void work(uint32_t slices, uint32_t rows_n, uint32_t wid, uint32_t warps,
                                         uint32_t* claimed) const {
        const uint32_t all = slices + (rows_n + kFanRows - 1u) / kFanRows, dealt = all / 8u * 7u / warps * warps;
        uint32_t ahead = 0u;
        auto after = [&](uint32_t i) {   // the item after i (dealt ones first)
            if (i + warps < dealt) return i + warps;
            const uint32_t c = __shfl_sync(kFull, ahead, 0);
            if (lane == 0) ahead = atomicAdd(claimed, 1u);
            return dealt + c;
        };
        auto fetch = [&](uint32_t i) {
            if (i < slices) return __ldcg(P.slices + i);
            const uint32_t r = (i - slices) * kFanRows + lane;
            return i < all && lane < kFanRows && r < rows_n ? __ldcg(P.rows + r) : make_uint4(0u, 0u, 0u, 0u);
        };
        if (lane == 0) ahead = atomicAdd(claimed, 1u);
        uint32_t i = wid < dealt ? wid : after(dealt);
        uint4 it = fetch(i);
        while (i < all) {
            const uint32_t i1 = after(i);
            const uint4 it1 = fetch(i1);
            if (i < slices) slice(it);
            else rows(it.x, it.y, (int32_t)it.z, (int32_t)(it.w - it.z));
            i = i1;
            it = it1;
        }
    }
};

// Barrier of the whole (cooperative) grid; `target`: arrivals so far.
__device__ __forceinline__ bool fan_barrier(FanSync* s, uint32_t target, unsigned long long deadline) {
    __syncthreads();
    int ok = 1;
    if (threadIdx.x == 0) {
        asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(&s->barrier.arrived) : "memory");
        for (uint32_t spins = 1; (int32_t)(ld_acquire(&s->barrier.arrived) - target) < 0; spins++)
            if ((spins & 1023u) == 0 && gtime() > deadline) {
                ok = 0;
                break;
            }
    }
    return __syncthreads_and(ok) != 0;
}

template <int WT, bool CORE>
__global__ void __launch_bounds__(kFanThreads, 1) fan_kernel(const __grid_constant__ FanParams P) {
    const uint32_t tid = threadIdx.x, lane = tid & 31u, gt = blockIdx.x * blockDim.x + tid;
    const uint32_t gn = gridDim.x * blockDim.x, wid = (tid >> 5) * gridDim.x + blockIdx.x, nw = gn >> 5;
    const unsigned long long deadline = gtime() + P.timeout_ns;
    // the group before gave up (set by an earlier kernel of the stream, so that
    // every block finds the same)
    if (ld_volatile_int(&P.ctrl->error) != kErrNone) return;
    const uint32_t places = P.mask + 1u;
    uint32_t arrivals = 0u;
    unsigned long long n_relax = 0ull;

    {
        const uint32_t inf = WT == 1 ? kInfF32 : kInfU32;
        const size_t rows = (size_t)P.n * 8u;
        for (size_t i = gt; i < rows; i += gn) {
            reinterpret_cast<uint4*>(P.dist)[i] = make_uint4(inf, inf, inf, inf);
            if (P.pred) reinterpret_cast<uint4*>(P.pred)[i] = make_uint4(kInfU32, kInfU32, kInfU32, kInfU32);
        }
        for (uint32_t i = gt; i < 2u * places; i += gn) P.wait[i] = 0u;
    }
    bool ok = fan_barrier(P.sync, arrivals += gridDim.x, deadline);
    if (ok && gt < (uint32_t)P.nq) {
        const uint32_t s = (uint32_t)P.srcs[gt];
        P.dist[(size_t)s * 32u + gt] = 0u;
        if (P.pred) P.pred[(size_t)s * 32u + gt] = s;
        atomicOr(P.wait + ((s * kWaveHash) & P.mask), 1u << gt);
    }
    ok = ok && fan_barrier(P.sync, arrivals += gridDim.x, deadline);

    uint32_t step = 0u;
    FanPass pass = CORE ? kFanCore : kFanRelax;
    bool deep = false;
    while (ok) {
        const uint32_t set = step & 3u;
        uint32_t* wait_r = P.wait + (size_t)(step & 1u) * places;
        uint32_t* wait_w = P.wait + (size_t)((step & 1u) ^ 1u) * places;
        // list the waiting vertices (all of them in the predecessor pass)
        for (uint32_t base = wid * 32u; base < places; base += nw * 32u) {
            const uint32_t v = ((base + lane) * kWaveHashInv) & P.mask;
            uint32_t m = 0u;
            int2 sp = make_int2(0, 0);
            if (base + lane < places) {
                if (pass == kFanTight || pass == kFanPull) {
                    if (v < (uint32_t)P.n) m = kFull;
                } else {
                    m = __ldcg(wait_r + base + lane);
                    if (m) wait_r[base + lane] = 0u;
                }
                if (m) sp = __ldg(P.span + v);
            }
            if (CORE && (pass == kFanCore || pass == kFanPull)) {
                // Eight rows at a time.  Core: the queries that wait below
                // their bound, and whether one of them is not at the core yet
                // and relaxes all arcs.  Pull: those that have not settled the
                // vertex; those that know a way there wait with it, as it has
                // relaxed nothing yet.
                const Fan<WT, kFanCore> f(P, nullptr);
                const int32_t deg = sp.y - sp.x;
                const bool has = deg > 0, hub = deg >= P.core_deg;
                const int32_t mid = has && pass == kFanCore ? __ldg(P.mid + v) : sp.y;
                const uint32_t row = min(v, (uint32_t)P.n - 1u), some = __ballot_sync(kFull, has);
                uint32_t open = 0u, told = 0u;
                for (int j0 = 0; j0 < 32; j0 += 8) {
                    if (!((some >> j0) & 255u)) continue;
                    uint32_t d[8];
#pragma unroll
                    for (int k = 0; k < 8; k++) {
                        const uint32_t off = f.at(__shfl_sync(kFull, row, j0 + k));
                        d[k] = (some >> (j0 + k)) & 1u ? __ldcg(f.word(P.dist, off)) : 0u;
                    }
#pragma unroll
                    for (int k = 0; k < 8; k++) {
                        const bool in = (__shfl_sync(kFull, m, j0 + k) >> lane) & 1u;
                        const bool core = __shfl_sync(kFull, (int)hub, j0 + k) != 0;
                        bool a, b;
                        if (pass == kFanCore) {
                            a = in && d[k] < f.bound;
                            b = a && d[k] < f.core;
                            if (b && core) atomicMax(P.sync->core + lane, ~d[k]);
                        } else {
                            a = in && f.core != kInfU32 && d[k] >= f.bound;
                            b = a && d[k] != Fan<WT, kFanCore>::kInf;
                        }
                        const uint32_t ma = __ballot_sync(kFull, a), mb = __ballot_sync(kFull, b);
                        if ((int)lane == j0 + k) open = ma, told = mb;
                    }
                }
                m = has ? open : 0u;
                if (pass == kFanCore) {
                    if (hub || !told) sp.y = mid;
                } else if (m && told && deg > 1) {
                    // (a vertex with one arc has nobody to tell but its source)
                    wait_w[base + lane] = told;
                }
                if (!m) sp.y = sp.x;
            }
            const int32_t deg = sp.y - sp.x;
            n_relax += (uint32_t)deg;
            const uint32_t sm = __ballot_sync(kFull, deg > 0 && deg <= kFanShort);
            uint32_t lm = __ballot_sync(kFull, deg > kFanShort);
            if (!(sm | lm)) continue;
            uint32_t k = deg > kFanShort ? ((uint32_t)deg + kFanChunk - 1u) / kFanChunk : 0u, incl = k;
            if (lm) {
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const uint32_t x = __shfl_up_sync(kFull, incl, o);
                    if (lane >= (uint32_t)o) incl += x;
                }
            }
            // lane 0 takes the room of the short rows, lane 31 that of the slices
            uint32_t at = 0u;
            if (lane == 0u && sm) at = atomicAdd(&P.sync->set[set].rows, (uint32_t)__popc(sm));
            if (lane == 31u && lm) at = atomicAdd(&P.sync->set[set].slices, incl);
            const uint32_t at_r = __shfl_sync(kFull, at, 0), at_s = __shfl_sync(kFull, at, 31) + incl - k;
            if ((sm >> lane) & 1u) P.rows[at_r + __popc(sm & lanemask_lt())] =
                    make_uint4(v, m, (uint32_t)sp.x, (uint32_t)sp.y);
            // one slice of its own row each, then the rest of the longest rows together
            if (k == 1u) P.slices[at_s] = make_uint4(v, m, (uint32_t)sp.x, (uint32_t)sp.y);
            lm = __ballot_sync(kFull, k > 1u);
            while (lm) {
                const int j = __ffs((int)lm) - 1;
                lm &= lm - 1u;
                const uint32_t vj = __shfl_sync(kFull, v, j), mj = __shfl_sync(kFull, m, j);
                const uint32_t kj = __shfl_sync(kFull, k, j), aj = __shfl_sync(kFull, at_s, j);
                const uint32_t b = (uint32_t)__shfl_sync(kFull, sp.x, j), e = (uint32_t)__shfl_sync(kFull, sp.y, j);
                for (uint32_t i = lane; i < kj; i += 32u) {
                    const uint32_t lo = b + i * kFanChunk;
                    P.slices[aj + i] = make_uint4(vj, mj, lo, min(e, lo + kFanChunk));
                }
            }
        }
        if (gt == 0) {
            const uint32_t z = (step + 2u) & 3u;
            P.sync->set[z].slices = P.sync->set[z].rows = P.sync->set[z].claimed = 0u;
        }
        if (!(ok = fan_barrier(P.sync, arrivals += gridDim.x, deadline))) break;
        const uint32_t slices = ld_relaxed(&P.sync->set[set].slices), rows = ld_relaxed(&P.sync->set[set].rows);
        if (pass == kFanTight) {
            Fan<WT, kFanTight>(P, wait_w).work(slices, rows, wid, nw, &P.sync->set[set].claimed);
            break;
        }
        if ((pass == kFanCore || pass == kFanRelax) && step >= P.max_steps) {
            deep = slices + rows > kFanTail || (slices + rows != 0u && step >= 16u * P.max_steps);
            if (deep) break;
        }
        if (slices + rows == 0u) {
            // nobody waits: the core has settled, or all distances are final
            if (CORE && pass == kFanCore) pass = kFanPull;
            else if (!P.pred) break;
            else pass = kFanTight;
        } else if (CORE && pass == kFanCore) {
            Fan<WT, kFanCore>(P, wait_w).work(slices, rows, wid, nw, &P.sync->set[set].claimed);
        } else if (CORE && pass == kFanPull) {
            Fan<WT, kFanPull>(P, wait_w).work(slices, rows, wid, nw, &P.sync->set[set].claimed);
            pass = kFanRelax;
        } else {
            Fan<WT, kFanRelax>(P, wait_w).work(slices, rows, wid, nw, &P.sync->set[set].claimed);
        }
        if (!(ok = fan_barrier(P.sync, arrivals += gridDim.x, deadline))) break;
        step++;
    }
    for (int o = 16; o > 0; o >>= 1) n_relax += __shfl_down_sync(kFull, n_relax, o);
    if (lane == 0 && n_relax) atomicAdd(&P.ctrl->stats[kStRelax], n_relax);
    if (tid == 0 && !ok) raise_error(P.ctrl, kErrTimeout, 22, 0);
    if (gt == 0) {
        atomicAdd(&P.ctrl->stats[kStIter], (unsigned long long)step);
        if (deep) raise_error(P.ctrl, kErrDeep, 23, (int)step);
        else atomicAdd(&P.ctrl->finished, P.nq);
    }
}

// Rows [n][32] -> the caller's [nq][n]: 32 x 32 tiles through shared memory.
static __global__ void __launch_bounds__(256) fan_out_kernel(const uint32_t* rows, int32_t n, int32_t nq, uint32_t* out) {
    __shared__ uint32_t tile[32][33];
    const uint32_t x = threadIdx.x & 31u, y = threadIdx.x >> 5;
    for (uint32_t v0 = blockIdx.x * 32u; v0 < (uint32_t)n; v0 += gridDim.x * 32u) {
#pragma unroll
        for (uint32_t k = 0; k < 32u; k += 8u)
            if (v0 + y + k < (uint32_t)n) tile[y + k][x] = __ldcg(rows + (size_t)(v0 + y + k) * 32u + x);
        __syncthreads();
#pragma unroll
        for (uint32_t k = 0; k < 32u; k += 8u)
            if (y + k < (uint32_t)nq && v0 + x < (uint32_t)n) out[(size_t)(y + k) * (uint32_t)n + v0 + x] = tile[x][y + k];
        __syncthreads();
    }
}

}  // namespace sssp
