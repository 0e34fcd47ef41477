// sssp_layout.cu -- the device layout of a graph: hubs split into shadow
// vertices, a second copy of the arcs of symmetric graphs with hubs whose rows
// have their light arcs first, and where every real vertex's arcs lie.  All of it runs on the device (built on
// the host, R-MAT-22's layout took 11 of the 17 ms of its creation).
#include <algorithm>
#include <cmath>
#include <cstring>

#include "../../include/sssp.h"
#include "api_internal.h"

namespace sssp {

namespace {

constexpr int kScanThreads = 256, kScanItems = 8, kScanTile = kScanThreads * kScanItems;
constexpr int32_t kBigRow = 2048;   // rows above this are copied and checked by a block, not a warp
constexpr int kBigThreads = 1024;

// Shadow vertices of a row and the arcs that move to them.  (Arc numbers and
// degrees end at 2^31 - 1: sums beyond a row are formed unsigned.)
__device__ __forceinline__ uint2 split_of(int32_t deg, int32_t split) {
    if (deg <= split) return make_uint2(0u, 0u);
    return make_uint2(((uint32_t)deg + (uint32_t)split - 1u) / (uint32_t)split, (uint32_t)deg);
}

__device__ __forceinline__ uint2 warp_scan(uint2 x, uint2& total) {   // inclusive
    const uint32_t lane = lane_id();
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t a = __shfl_up_sync(kFull, x.x, o), b = __shfl_up_sync(kFull, x.y, o);
        if (lane >= (uint32_t)o) {
            x.x += a;
            x.y += b;
        }
    }
    total = make_uint2(__shfl_sync(kFull, x.x, 31), __shfl_sync(kFull, x.y, 31));
    return x;
}

// Exclusive block scan (blockDim.x a multiple of 32, at most 1024).
__device__ uint2 block_scan(uint2 x, uint2& total) {
    __shared__ uint2 part[33];
    const uint32_t lane = lane_id(), w = threadIdx.x >> 5, nw = blockDim.x >> 5;
    uint2 wt;
    const uint2 incl = warp_scan(x, wt);
    if (lane == 0) part[w] = wt;
    __syncthreads();
    if (w == 0) {
        uint2 t = lane < nw ? part[lane] : make_uint2(0u, 0u), all;
        const uint2 i = warp_scan(t, all);
        if (lane < nw) part[lane] = make_uint2(i.x - t.x, i.y - t.y);
        if (lane == 0) part[32] = all;
    }
    __syncthreads();
    total = part[32];
    const uint2 base = part[w];
    __syncthreads();
    return make_uint2(base.x + incl.x - x.x, base.y + incl.y - x.y);
}

__global__ void __launch_bounds__(kScanThreads) split_sums_kernel(const int32_t* rp, int32_t n, int32_t split,
                                                                  uint2* sums) {
    uint2 x = make_uint2(0u, 0u), total;
    const int64_t base = (int64_t)blockIdx.x * kScanTile;
    for (int i = 0; i < kScanItems; i++) {
        const int64_t v = base + i * kScanThreads + threadIdx.x;
        if (v < n) {
            const uint2 k = split_of(rp[v + 1] - rp[v], split);
            x.x += k.x;
            x.y += k.y;
        }
    }
    block_scan(x, total);
    if (threadIdx.x == 0) sums[blockIdx.x] = total;
}

// Exclusive scan of the tiles' sums, their total at sums[tiles].  One block.
__global__ void __launch_bounds__(1024) split_scan_kernel(uint2* sums, int tiles) {
    uint2 run = make_uint2(0u, 0u);
    for (int b = 0; b < tiles; b += 1024) {
        const int i = b + (int)threadIdx.x;
        uint2 total;
        const uint2 ex = block_scan(i < tiles ? sums[i] : make_uint2(0u, 0u), total);
        if (i < tiles) sums[i] = make_uint2(run.x + ex.x, run.y + ex.y);
        run.x += total.x;
        run.y += total.y;
    }
    if (threadIdx.x == 0) sums[tiles] = run;
}

// Row offsets of the split layout: real vertices first (a hub's row links its
// shadows), then the shadows in vertex order; first[v] = a hub's first shadow
// or -1.  at0 (or null): where row v lies without the links, hubs last.
__global__ void __launch_bounds__(kScanThreads) split_rows_kernel(const int32_t* rp, int32_t n, int64_t m,
                                                                  int32_t split, const uint2* sums, int tiles,
                                                                  int32_t* rp1, int32_t* first, int32_t* owner,
                                                                  int32_t* at0) {
    const uint2 all = sums[tiles];
    const int64_t shadows0 = m - (int64_t)all.y + (int64_t)all.x;   // where the shadows' arcs begin
    const int64_t base = (int64_t)blockIdx.x * kScanTile + (int64_t)threadIdx.x * kScanItems;
    uint2 x = make_uint2(0u, 0u), total;
    for (int i = 0; i < kScanItems; i++)
        if (base + i < n) {
            const uint2 k = split_of(rp[base + i + 1] - rp[base + i], split);
            x.x += k.x;
            x.y += k.y;
        }
    uint2 at = block_scan(x, total);
    at.x += sums[blockIdx.x].x;
    at.y += sums[blockIdx.x].y;
    for (int i = 0; i < kScanItems; i++) {
        const int64_t v = base + i;
        if (v >= n) break;
        const uint2 k = split_of(rp[v + 1] - rp[v], split);
        rp1[v] = (int32_t)((int64_t)rp[v] - at.y + at.x);
        first[v] = k.x ? (int32_t)(n + (int64_t)at.x) : -1;
        if (at0) at0[v] = (int32_t)(k.x ? m - (int64_t)all.y + at.y : (int64_t)rp[v] - at.y);
        for (uint32_t j = 0; j < k.x; j++) {
            owner[at.x + j] = (int32_t)v;
            rp1[(int64_t)n + at.x + j] = (int32_t)(shadows0 + at.y + (int64_t)j * split);
        }
        at.x += k.x;
        at.y += k.y;
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) rp1[(int64_t)n + all.x] = (int32_t)(m + (int64_t)all.x);
}

// Copies `count` arcs by one warp, those of weight <= light first (both parts
// in order).
__device__ void part_row_warp(const uint2* from, uint2* to, int32_t count, uint32_t light) {
    const uint32_t lane = lane_id();
    int32_t nl = 0;
    for (int32_t b = 0; b < count; b += 32)
        nl += __popc(__ballot_sync(kFull, b + (int32_t)lane < count && from[b + lane].y <= light));
    int32_t l = 0, h = nl;
    for (int32_t b = 0; b < count; b += 32) {
        const bool in = b + (int32_t)lane < count;
        const uint2 a = in ? from[b + lane] : make_uint2(0u, 0u);
        const uint32_t lm = __ballot_sync(kFull, in && a.y <= light), hm = __ballot_sync(kFull, in && a.y > light);
        if (in) to[a.y <= light ? l + __popc(lm & lanemask_lt()) : h + __popc(hm & lanemask_lt())] = a;
        l += __popc(lm);
        h += __popc(hm);
    }
}

// Row v of the original arrays (rp0, adj0) and of the split layout (rp1, first, adj1).
__device__ __forceinline__ int32_t split_at(const int32_t* rp1, const int32_t* first, int64_t v) {
    return first[v] >= 0 ? rp1[first[v]] : rp1[v];
}

// The rows to their places in the split layout and the links of every hub, one
// warp per vertex; rows above kBigRow arcs by the next kernel.
__global__ void relayout_kernel(const int32_t* rp0, const uint2* adj0, int32_t n, const int32_t* rp1,
                                const int32_t* first, int32_t split, uint2* adj1) {
    const int64_t wid = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    const uint32_t lane = lane_id();
    for (int64_t v = wid; v < n; v += nw) {
        const int32_t b = rp0[v], deg = rp0[v + 1] - b, s0 = first[v];
        if (s0 >= 0) {
            const int32_t k = (int32_t)split_of(deg, split).x, at = rp1[v];
            for (int32_t j = (int32_t)lane; j < k; j += 32) adj1[at + j] = make_uint2((uint32_t)(s0 + j), 0u);
        }
        if (deg > kBigRow) continue;
        const int32_t to = split_at(rp1, first, v);
        for (int32_t j = (int32_t)lane; j < deg; j += 32) adj1[to + j] = adj0[b + j];
    }
}

// Light-first rows out of the split layout, at their places at0.
__global__ void light_first_kernel(const int32_t* rp0, uint2* adj0, int32_t n, const int32_t* rp1,
                                   const int32_t* first, const int32_t* at0, uint32_t light, const uint2* adj1) {
    const int64_t wid = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t v = wid; v < n; v += nw) {
        const int32_t deg = rp0[v + 1] - rp0[v];
        if (deg > 0 && deg <= kBigRow) part_row_warp(adj1 + split_at(rp1, first, v), adj0 + at0[v], deg, light);
    }
}

// The rows above kBigRow arcs of the two kernels above, one block per vertex.
template <bool LIGHT_FIRST>
__global__ void __launch_bounds__(kBigThreads) relayout_big_kernel(const int32_t* rp0, uint2* adj0, int32_t n,
                                                                   const int32_t* rp1, const int32_t* first,
                                                                   const int32_t* at0, uint32_t light, uint2* adj1) {
    __shared__ int32_t list[kBigThreads];
    __shared__ int listed;
    const int64_t step = (int64_t)gridDim.x * kBigThreads;
    for (int64_t base = (int64_t)blockIdx.x * kBigThreads; base < n; base += step) {
        if (threadIdx.x == 0) listed = 0;
        __syncthreads();
        const int64_t v = base + threadIdx.x;
        if (v < n && rp0[v + 1] - rp0[v] > kBigRow) list[atomicAdd(&listed, 1)] = (int32_t)v;
        __syncthreads();
        for (int i = 0; i < listed; i++) {
            const int32_t u = list[i];
            const uint32_t deg = (uint32_t)(rp0[u + 1] - rp0[u]);
            uint2 *row0 = adj0 + (LIGHT_FIRST ? at0[u] : rp0[u]), *row1 = adj1 + split_at(rp1, first, u);
            if (!LIGHT_FIRST) {
                for (uint32_t e = threadIdx.x; e < deg; e += kBigThreads) row1[e] = row0[e];
                continue;
            }
            uint2 mine = make_uint2(0u, 0u), total;
            for (uint32_t e = threadIdx.x; e < deg; e += kBigThreads) mine.x += row1[e].y <= light;
            block_scan(mine, total);
            uint32_t l = 0u, h = total.x;
            for (uint32_t e0 = 0; e0 < deg; e0 += kBigThreads) {
                const uint32_t e = e0 + threadIdx.x;
                const bool in = e < deg;
                const uint2 a = in ? row1[e] : make_uint2(0u, 0u);
                const bool lt = in && a.y <= light;
                uint2 tile;
                const uint2 at = block_scan(make_uint2(lt, in && !lt), tile);
                if (in) row0[lt ? l + at.x : h + at.y] = a;
                l += tile.x;
                h += tile.y;
            }
        }
        __syncthreads();
    }
}

// Where the arcs of every real vertex lie: its row, or (a split hub, whose row
// links its shadows) the shadows' rows, which follow one another; with at0, rows
// of these lengths from at0[v] on.  mid (with at0): the end of the light arcs;
// their count is added to *lights.
__global__ void span_kernel(const int32_t* rp, const uint2* adj, int32_t n, int2* span, const int32_t* at0,
                            uint32_t light, int32_t* mid, unsigned long long* lights) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    unsigned long long count = 0;
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += stride) {
        int32_t b = rp[v], e = rp[v + 1];
        if (at0) {
            e = at0[v] + (e - b);
            b = at0[v];
        } else if (e > b) {
            const uint32_t first = adj[b].x;
            if (first >= (uint32_t)n) {
                const int32_t k = e - b;
                b = rp[first];
                e = rp[first + (uint32_t)k];
            }
        }
        span[v] = make_int2(b, e);
        if (mid) {
            int32_t lo = b, hi = e;   // the first heavy arc
            while (lo < hi) {
                const int32_t c = lo + (hi - lo) / 2;
                if (adj[c].y <= light) lo = c + 1;
                else hi = c;
            }
            mid[v] = lo;
            count += (unsigned long long)(lo - b);
        }
    }
    if (!mid) return;
    for (int o = 16; o > 0; o >>= 1) count += __shfl_down_sync(kFull, count, o);
    if (lane_id() == 0 && count) atomicAdd(lights, count);
}

// The first four arcs of every vertex at a fixed place.
__global__ void quads_kernel(const int2* span, const uint2* adj, int32_t n, uint4* quads) {
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t v = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; v < n; v += stride) {
        const int2 sp = span[v];
        uint2 a[4];
#pragma unroll
        for (int k = 0; k < 4; k++) a[k] = k < sp.y - sp.x ? adj[sp.x + k] : make_uint2(kNoArc, 0u);
        if (sp.y - sp.x > 4) a[0].x |= 0x80000000u;
        quads[2 * v] = make_uint4(a[0].x, a[0].y, a[1].x, a[1].y);
        quads[2 * v + 1] = make_uint4(a[2].x, a[2].y, a[3].x, a[3].y);
    }
}

// Original arc order from a split layout: the arcs of vertex v lie from
// src_start[v] on.  One warp per vertex.
__global__ void unsplit_kernel(const uint2* adj1, const int32_t* src_start, const int32_t* rp0, int32_t n,
                               uint2* adj0) {
    const int64_t wid = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    const uint32_t lane = lane_id();
    for (int64_t v = wid; v < n; v += nw) {
        const int32_t b = rp0[v], e = rp0[v + 1], src = src_start[v];
        for (int32_t i = (int32_t)lane; i < e - b; i += 32) adj0[b + i] = adj1[src + i];
    }
}

// Symmetry, shown arc by arc on rows of strictly increasing columns.  Of the
// two directions of an edge, the one from the vertex of more arcs (or, of
// equally many, the smaller number) is looked up in the other's row, the
// shorter one; the lookups and the arcs of the other kind must be as many.
struct SymState {
    int bad, pad;
    unsigned long long looked, other;
};

__device__ __forceinline__ void check_arc(const int32_t* rp, const uint2* adj, int32_t u, int32_t du, int32_t first,
                                          uint32_t e, int& bad, unsigned long long& looked,
                                          unsigned long long& other) {
    const uint2 a = adj[e];
    if (e > (uint32_t)first && adj[e - 1u].x >= a.x) bad = 1;
    const int32_t v = (int32_t)a.x;
    if (v == u) return;
    int32_t lo = rp[v], hi = rp[v + 1];
    const int32_t dv = hi - lo;
    if (dv > du || (dv == du && v < u)) {
        other++;
        return;
    }
    looked++;
    const int32_t end = hi;
    while (lo < hi) {
        const int32_t c = lo + (hi - lo) / 2;
        if (adj[c].x < (uint32_t)u) lo = c + 1;
        else hi = c;
    }
    if (lo >= end || adj[lo].x != (uint32_t)u || adj[lo].y != a.y) bad = 1;
}

__device__ __forceinline__ void sym_publish(SymState* st, int bad, unsigned long long looked,
                                            unsigned long long other) {
    bad = __any_sync(kFull, bad);
    for (int o = 16; o > 0; o >>= 1) {
        looked += __shfl_down_sync(kFull, looked, o);
        other += __shfl_down_sync(kFull, other, o);
    }
    if (lane_id() == 0) {
        if (bad) atomicOr(&st->bad, 1);
        if (looked) atomicAdd(&st->looked, looked);
        if (other) atomicAdd(&st->other, other);
    }
}

__global__ void symmetry_kernel(const int32_t* rp, const uint2* adj, int32_t n, SymState* st) {
    const int64_t wid = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    const uint32_t lane = lane_id();
    unsigned long long looked = 0, other = 0;
    int bad = 0, k = 0;
    for (int64_t v = wid; v < n; v += nw) {
        // a directed graph is recognised by its first rows
        if ((k++ & 31) == 0 && __any_sync(kFull, bad || ld_volatile_int(&st->bad))) {
            bad = 1;
            break;
        }
        const int32_t b = rp[v], e = rp[v + 1];
        if (e - b > kBigRow) continue;
        for (uint32_t i = (uint32_t)b + lane; i < (uint32_t)e; i += 32u)
            check_arc(rp, adj, (int32_t)v, e - b, b, i, bad, looked, other);
        __syncwarp();
    }
    sym_publish(st, bad, looked, other);
}

__global__ void __launch_bounds__(kBigThreads) symmetry_big_kernel(const int32_t* rp, const uint2* adj, int32_t n,
                                                                   SymState* st) {
    __shared__ int32_t list[kBigThreads];
    __shared__ int listed;
    const int64_t step = (int64_t)gridDim.x * kBigThreads;
    unsigned long long looked = 0, other = 0;
    int bad = 0;
    for (int64_t base = (int64_t)blockIdx.x * kBigThreads; base < n; base += step) {
        if (threadIdx.x == 0) listed = 0;
        __syncthreads();
        const int64_t v = base + threadIdx.x;
        if (v < n && rp[v + 1] - rp[v] > kBigRow) list[atomicAdd(&listed, 1)] = (int32_t)v;
        __syncthreads();
        for (int i = 0; i < listed; i++) {
            const int32_t u = list[i], b = rp[u], e = rp[u + 1];
            for (uint32_t j = (uint32_t)b + threadIdx.x; j < (uint32_t)e; j += kBigThreads)
                check_arc(rp, adj, u, e - b, b, j, bad, looked, other);
        }
        __syncthreads();
    }
    sym_publish(st, bad, looked, other);
}

int warps_grid(const Graph* g) { return g->sms * 8; }
int span_grid(const Graph* g) {
    return (int)std::max<int64_t>(1, std::min<int64_t>(((int64_t)g->n + 255) / 256, (int64_t)g->sms * 8));
}

}  // namespace

int check_symmetry(Graph* g, const int32_t* rp0, const uint2* adj0, cudaStream_t s) {
    g->symmetric = false;
    // hubs are what light-first rows pay for
    if (g->feat.max_deg <= 512.0 || g->m < (1 << 18)) return SSSP_OK;
    SymState* st = nullptr;
    SymState h;
    if (cudaMalloc((void**)&st, sizeof(SymState)) != cudaSuccess) {
        cudaGetLastError();
        return SSSP_E_NOMEM;
    }
    cudaMemsetAsync(st, 0, sizeof(SymState), s);
    symmetry_kernel<<<warps_grid(g), 256, 0, s>>>(rp0, adj0, g->n, st);
    symmetry_big_kernel<<<g->sms, kBigThreads, 0, s>>>(rp0, adj0, g->n, st);
    cudaMemcpyAsync(&h, st, sizeof(h), cudaMemcpyDeviceToHost, s);
    const cudaError_t e = cudaStreamSynchronize(s);
    cudaFree(st);
    if (e != cudaSuccess) return cuda_status(e);
    g->symmetric = h.bad == 0 && h.looked == h.other;
    // A seventh of the average weight: a fourteenth of the arcs of evenly
    // distributed weights; of small whole weights a few values.  us at a
    // quarter, sixth, eighth and tenth: R-MAT-22 665, 636, 638, 672; R-MAT-20
    // 311, 274, 263, 262; R-MAT-19 f32 311, 286, 272, 264; 64 queries on
    // R-MAT-20 4100, 3740, 3780, 4940 (too few settle), on R-MAT-18 f32 2670,
    // 2560, 2400, 2320.
    const double lw = g->feat.avg_w / 7.0;
    g->light_w = g->wtype == SSSP_W_F32 ? __float_as_uint_host((float)lw) : (uint32_t)std::max(3.0, std::floor(lw));
    return SSSP_OK;
}

void launch_unsplit(const Graph* g, const int32_t* src_start, const int32_t* rp0, uint2* adj0, cudaStream_t s) {
    unsplit_kernel<<<warps_grid(g), 256, 0, s>>>(g->adj, src_start, rp0, g->n, adj0);
}

// The arcs of a symmetric graph with hubs once more, light arcs first, in the
// array of the original ones (adj0; hubs last: with them in between, 64 queries on
// R-MAT-18 f32 took 1 to 3% longer), for the wavefront kernels; span and mid describe
// them from now on, in every layout.  The queue engine keeps the original order:
// with rows partitioned for both it relaxed 43% more arcs (a hub's slices were
// all light or all heavy), R-MAT-20 1.41 ms -> 1.89, R-MAT-18 1.03 -> 1.29.
// They only save time: without room, false.
static bool light_first(Graph* g, const int32_t* rp0, uint2* adj0, const int32_t* rp1, const int32_t* first,
                        const int32_t* at0, uint2* adj1, cudaStream_t s) {
    const int32_t n = g->n;
    unsigned long long *lights = nullptr, h = 0;
    int32_t* mid = nullptr;
    if ((!g->span && cudaMalloc((void**)&g->span, sizeof(int2) * (size_t)n) != cudaSuccess) ||
        cudaMalloc((void**)&mid, sizeof(int32_t) * (size_t)n) != cudaSuccess ||
        cudaMalloc((void**)&lights, sizeof(*lights)) != cudaSuccess) {
        cudaGetLastError();
        cudaFree(mid);
        return false;
    }
    light_first_kernel<<<warps_grid(g), 256, 0, s>>>(rp0, adj0, n, rp1, first, at0, g->light_w, adj1);
    relayout_big_kernel<true><<<g->sms, kBigThreads, 0, s>>>(rp0, adj0, n, rp1, first, at0, g->light_w, adj1);
    cudaMemsetAsync(lights, 0, sizeof(*lights), s);
    span_kernel<<<span_grid(g), 256, 0, s>>>(rp0, adj0, n, g->span, at0, g->light_w, mid, lights);
    cudaMemcpyAsync(&h, lights, sizeof(h), cudaMemcpyDeviceToHost, s);
    const bool ok = cudaStreamSynchronize(s) == cudaSuccess;
    cudaFree(lights);
    if (!ok) {
        cudaFree(mid);
        return false;
    }
    g->wadj = adj0;
    g->mid = mid;
    g->light_share = (double)h / (double)g->m;
    return true;
}

int build_layout(Graph* g, int32_t* rp0, uint2* adj0, int32_t split, cudaStream_t s) {
    const int32_t n = g->n;
    const int tiles = (int)(((int64_t)n + kScanTile - 1) / kScanTile);
    uint2* sums = nullptr;
    uint2 all = make_uint2(0u, 0u);
    if (g->feat.max_deg > (double)split) {
        if (cudaMalloc((void**)&sums, sizeof(uint2) * ((size_t)tiles + 1)) != cudaSuccess) {
            cudaGetLastError();
            return SSSP_E_NOMEM;
        }
        split_sums_kernel<<<tiles, kScanThreads, 0, s>>>(rp0, n, split, sums);
        split_scan_kernel<<<1, 1024, 0, s>>>(sums, tiles);
        cudaMemcpyAsync(&all, sums + tiles, sizeof(all), cudaMemcpyDeviceToHost, s);
        const cudaError_t e = cudaStreamSynchronize(s);
        if (e != cudaSuccess) {
            cudaFree(sums);
            return cuda_status(e);
        }
    }
    const int64_t ns = all.x;
    if (ns == 0 || (int64_t)n + ns > 2147483647LL || g->m + ns > 2147483647LL) {
        cudaFree(sums);
        g->row_ptr = rp0;
        g->adj = adj0;
        g->owner = nullptr;
        g->nv = n;
        g->mv = g->m;
        g->split = 0;
        return SSSP_OK;
    }
    const int32_t nv = (int32_t)(n + ns);
    const int64_t mv = g->m + ns;   // every hub's arcs move, and a link per shadow comes
    int32_t *rp1 = nullptr, *first = nullptr, *owner = nullptr, *at0 = nullptr;
    uint2* adj1 = nullptr;
    int rc = SSSP_OK;
    if (cudaMalloc((void**)&rp1, sizeof(int32_t) * ((size_t)nv + 1)) != cudaSuccess ||
        cudaMalloc((void**)&first, sizeof(int32_t) * (size_t)n) != cudaSuccess ||
        cudaMalloc((void**)&owner, sizeof(int32_t) * (size_t)ns) != cudaSuccess ||
        cudaMalloc((void**)&adj1, sizeof(uint2) * (size_t)mv) != cudaSuccess) {
        cudaGetLastError();
        rc = SSSP_E_NOMEM;
    }
    if (rc == SSSP_OK) {
        if (g->symmetric && !g->wadj && cudaMalloc((void**)&at0, sizeof(int32_t) * (size_t)n) != cudaSuccess) {
            cudaGetLastError();   // (only saves time)
            at0 = nullptr;
        }
        split_rows_kernel<<<tiles, kScanThreads, 0, s>>>(rp0, n, g->m, split, sums, tiles, rp1, first, owner, at0);
        relayout_kernel<<<warps_grid(g), 256, 0, s>>>(rp0, adj0, n, rp1, first, split, adj1);
        relayout_big_kernel<false><<<g->sms, kBigThreads, 0, s>>>(rp0, adj0, n, rp1, first, nullptr, 0u, adj1);
        if (cudaStreamSynchronize(s) != cudaSuccess) rc = SSSP_E_CUDA;
    }
    const bool keep = rc == SSSP_OK && at0 && light_first(g, rp0, adj0, rp1, first, at0, adj1, s);
    cudaFree(at0);
    cudaFree(sums);
    cudaFree(first);
    if (rc != SSSP_OK) {
        cudaFree(rp1);
        cudaFree(owner);
        cudaFree(adj1);
        return rc;
    }
    cudaFree(rp0);
    if (!keep) cudaFree(adj0);
    g->row_ptr = rp1;
    g->adj = adj1;
    g->owner = owner;
    g->nv = nv;
    g->mv = mv;
    g->split = split;
    return SSSP_OK;
}

int fill_span(Graph* g, cudaStream_t s) {
    if (g->wadj) return SSSP_OK;   // light_first has filled it
    if (!g->span && cudaMalloc((void**)&g->span, sizeof(int2) * (size_t)g->n) != cudaSuccess) {
        cudaGetLastError();
        return SSSP_E_NOMEM;
    }
    span_kernel<<<span_grid(g), 256, 0, s>>>(g->row_ptr, g->adj, g->n, g->span, nullptr, 0u, nullptr, nullptr);
    if (thin_graph(g->feat.avg_deg, g->feat.max_deg)) {
        if (!g->quads && cudaMalloc((void**)&g->quads, 2 * sizeof(uint4) * (size_t)g->n) != cudaSuccess) {
            // they only save time: without room for them, without them
            cudaGetLastError();
            g->quads = nullptr;
        }
        if (g->quads) quads_kernel<<<span_grid(g), 256, 0, s>>>(g->span, g->adj, g->n, g->quads);
    }
    return cuda_status(cudaStreamSynchronize(s));
}

}  // namespace sssp
