// sssp_noalloc.cu -- a single-source solve that allocates no memory.
//
// Some callers cannot allocate device memory at the time they want a
// shortest-path answer: code running under a memory pool or arena that owns
// every allocation of the process, plugins or real-time loops whose
// allocation budget is fixed up front, and code that must not call
// cudaMalloc/cudaFree because those calls can synchronise the device.  The
// regular entry points create a graph handle and a per-graph workspace; this
// one runs the wavefront kernels (wave.cuh) with all of their scratch state
// (control block, pending bits, hub slices, packed distance/predecessor
// words) in one fixed-size array that is part of the library image.  On
// R-MAT-13 with predecessors (GB300) a call takes 190 us; through the
// queues, with rings in the same array, it took 1600, and a graph whose front
// outgrew the rings failed.
//
// The array is a file-scope __device__ variable: every GPU that loads the
// library holds it (kNoAllocBytes, about 26 MiB) until the process exits.
// Host code cannot use the array's name as a device address, so the first
// call on each device resolves it with cudaGetSymbolAddress (with that device
// current).  All calls share the array and it keeps the previous call's
// contents: every call first re-initialises what must start empty (the
// control block, the pending bits, the distance words), so no call depends on
// how the previous one ended.  Calls that overlap on the GPU
// would race on the array; this file serialises the calls it issues with a
// process-wide mutex and returns only after the GPU work has finished.  A
// call reads results back and synchronises its stream part-way, so it must
// not be issued on a stream that is being captured into a CUDA graph.
#include <algorithm>
#include <cstring>
#include <mutex>

#include "../../include/sssp.h"
#include "internal.h"
#include "wave.h"

namespace sssp {

namespace {

constexpr size_t kCtrlBytes = 4096;
constexpr size_t kFlagBytes = 256;
constexpr size_t kSyncBytes = sizeof(TideSync);
constexpr size_t kBitBytes = 4 * sizeof(uint32_t) << kTideLogWords;       // near[2], far[2] of the grid kernel
constexpr size_t kItemBytes = (size_t)8 << 20;                            // its hub slices, two lists
constexpr size_t kWorkBytes = (size_t)SSSP_NOALLOC_MAX_VERTICES * sizeof(unsigned long long);
constexpr size_t kNoAllocBytes = kCtrlBytes + kFlagBytes + kSyncBytes + kBitBytes + kItemBytes + kWorkBytes;

// up to 2^17 words of 32 bits the grid kernel takes 2^17 words or fewer
static_assert((size_t)SSSP_NOALLOC_MAX_VERTICES <= (size_t)32 << kTideLogWords, "pending bits do not fit");
static_assert(sizeof(Ctrl) <= kCtrlBytes, "control block does not fit");

// The scratch array.  Device code could name it directly; host code only
// ever uses the address returned by cudaGetSymbolAddress.
static __device__ __align__(256) unsigned char g_noalloc_scratch[kNoAllocBytes];

// Validation flags and graph statistics for the launch shape.
struct NaFlags {
    int bad;                  // bit 0 row_ptr, bit 1 column range, bit 2 f32 weight
    unsigned int min_not;     // complement of the smallest weight (u32 value or f32 bits)
    unsigned int max_deg;
    unsigned int pad;
    double sum_w;
};

// Checks the row offsets and the interleaved (column, weight) arcs, and
// gathers the smallest weight, their sum (for the predecessor rule and the
// threshold step) and the largest degree.
__global__ void na_check_kernel(const int32_t* row_ptr, const uint2* arcs, int32_t n, int64_t m, int f32,
                                NaFlags* fl) {
    const int64_t first = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    unsigned int mn = 0xffffffffu, md = 0u;
    double sw = 0.0;
    int bad = 0;
    for (int64_t i = first; i <= n; i += stride) {
        const int32_t r = row_ptr[i], e = i < n ? row_ptr[i + 1] : r;
        if ((i == 0 && r != 0) || (i == n && (int64_t)r != m) || r < 0 || (int64_t)r > m || e < r) bad |= 1;
        else md = max(md, (unsigned int)(e - r));
    }
    for (int64_t i = first; i < m; i += stride) {
        const uint2 a = arcs[i];
        if ((int32_t)a.x < 0 || (int32_t)a.x >= n) bad |= 2;
        uint32_t wb = a.y;
        if (f32) {
            if (wb == 0x80000000u) wb = 0u;  // -0.0 adds like +0.0
            if ((wb & 0x80000000u) || (wb & 0x7f800000u) == 0x7f800000u) bad |= 4;
            sw += (double)__uint_as_float(wb);
        } else {
            sw += (double)wb;
        }
        mn = min(mn, wb);
    }
    for (int o = 16; o > 0; o >>= 1) {
        sw += __shfl_down_sync(kFull, sw, o);
        mn = min(mn, __shfl_down_sync(kFull, mn, o));
        md = max(md, __shfl_down_sync(kFull, md, o));
        bad |= __shfl_down_sync(kFull, bad, o);
    }
    if ((threadIdx.x & 31u) == 0) {
        if (bad) atomicOr(&fl->bad, bad);
        atomicMax(&fl->min_not, ~mn);
        atomicMax(&fl->max_deg, md);
        if (sw != 0.0) atomicAdd(&fl->sum_w, sw);
    }
}

struct NaDevice {
    bool ready = false;
    unsigned char* base = nullptr;   // device address of g_noalloc_scratch
};

std::mutex g_na_mu;
NaDevice g_na_dev[64];

struct NaLayout {
    Ctrl* ctrl;
    NaFlags* flags;
    TideSync* sync;
    uint32_t* bits;
    uint4* items;
    unsigned long long* work;
};

NaLayout na_layout(unsigned char* base) {
    NaLayout L;
    unsigned char* p = base;
    L.ctrl = reinterpret_cast<Ctrl*>(p);
    p += kCtrlBytes;
    L.flags = reinterpret_cast<NaFlags*>(p);
    p += kFlagBytes;
    L.sync = reinterpret_cast<TideSync*>(p);
    p += kSyncBytes;
    L.bits = reinterpret_cast<uint32_t*>(p);
    p += kBitBytes;
    L.items = reinterpret_cast<uint4*>(p);
    p += kItemBytes;
    L.work = reinterpret_cast<unsigned long long*>(p);
    return L;
}

bool device_memory(const void* p) {
    cudaPointerAttributes a;
    if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged;
}

}  // namespace
}  // namespace sssp

using namespace sssp;

extern "C" int sssp_solve_noalloc(const int32_t* row_ptr, const uint32_t* arcs, int32_t n, int64_t m,
                                  int32_t wtype, int32_t src, void* dist_out, int32_t* pred_out,
                                  void* stream_ptr) {
    if (!row_ptr || !dist_out || (m > 0 && !arcs)) return SSSP_E_INVAL;
    if (n < 1 || n > SSSP_NOALLOC_MAX_VERTICES || m < 0 || m > 2147483647LL) return SSSP_E_INVAL;
    if (wtype != SSSP_W_U32 && wtype != SSSP_W_F32) return SSSP_E_INVAL;
    if (src < 0 || src >= n) return SSSP_E_INVAL;
    if (!device_memory(row_ptr) || !device_memory(dist_out) || (m > 0 && !device_memory(arcs)) ||
        (pred_out && !device_memory(pred_out)))
        return SSSP_E_INVAL;
    cudaStream_t stream = (cudaStream_t)stream_ptr;
    std::lock_guard<std::mutex> lk(g_na_mu);
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return SSSP_E_CUDA;
    int sms = 0;
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    NaDevice& D = g_na_dev[dev];
    if (!D.ready) {
        // once per device, with this device current: the array's device address
        void* ptr = nullptr;
        if (cudaGetSymbolAddress(&ptr, g_noalloc_scratch) != cudaSuccess || !ptr) {
            cudaGetLastError();
            return SSSP_E_CUDA;
        }
        D.base = static_cast<unsigned char*>(ptr);
        D.ready = true;
    }
    NaLayout L = na_layout(D.base);
    const bool f32 = wtype == SSSP_W_F32;

    // validate the CSR (a bad column would make the kernel touch memory out of range)
    NaFlags hf;
    std::memset(&hf, 0, sizeof(hf));
    cudaMemsetAsync(L.ctrl, 0, kCtrlBytes + kFlagBytes + kSyncBytes, stream);
    const int64_t most = std::max<int64_t>((int64_t)n + 1, m);
    const int blocks = (int)std::max<int64_t>(1, std::min<int64_t>((most + 255) / 256, (int64_t)sms * 8));
    na_check_kernel<<<blocks, 256, 0, stream>>>(row_ptr, reinterpret_cast<const uint2*>(arcs), n, m, f32 ? 1 : 0,
                                                L.flags);
    if (cudaMemcpyAsync(&hf, L.flags, sizeof(hf), cudaMemcpyDeviceToHost, stream) != cudaSuccess ||
        cudaStreamSynchronize(stream) != cudaSuccess)
        return SSSP_E_CUDA;
    if (hf.bad) return SSSP_E_BADGRAPH;

    const int pred_mode = pred_out ? ((!f32 && m > 0 && ~hf.min_not >= 1u) ? 1 : 2) : 0;
    const double avg_w = m > 0 ? hf.sum_w / (double)m : 1.0;
    WaveGraph wg{n, m, avg_w, (double)hf.max_deg, sms, false, false, false, false, 0};
    Ctrl hc;
    bool clusters = true;
    for (;;) {
        WavePlan plan;
        plan_wave(wg, 1, pred_mode, &plan);
        if (!clusters) {
            plan.kind = kWholeGrid;
            plan.log_g = 0;
            plan.threads = 1024;
        }
        WaveParams P;
        std::memset(&P, 0, sizeof(P));
        const size_t smem = wave_params(plan, wg, f32, false, &P);
        P.row = row_ptr;
        P.adj = reinterpret_cast<const uint2*>(arcs);
        P.src0 = src;
        P.work = pred_mode ? (void*)L.work : dist_out;
        P.dist_out = (uint32_t*)dist_out;
        P.pred_out = pred_out;
        P.ctrl = L.ctrl;
        P.sync = L.sync;
        P.bits = L.bits;
        P.items = L.items;
        P.items_cap = (uint32_t)(kItemBytes / sizeof(uint4) / 2);
        // more slices than the lists hold: hubs are left to their warps
        if (tide_slices(m, P.hub_deg) > P.items_cap) P.has_hubs = 0;
        const bool grid = plan.kind == kWholeGrid;
        if (grid ? (size_t)P.words * 4 * sizeof(uint32_t) > kBitBytes : smem > kWaveMaxShared) return SSSP_E_INVAL;
        GridTurn turn(dev);
        if (grid) turn.wait();
        const cudaError_t ce = grid ? launch_tide(f32 ? 1 : 0, pred_mode, P, sms, plan.threads, stream)
                                    : launch_wave(f32 ? 1 : 0, pred_mode, P, 1, plan.threads, smem, stream);
        if (ce != cudaSuccess && !grid) {
            // no room for a cluster on this device (a part of one): the grid needs none
            cudaGetLastError();
            clusters = false;
            continue;
        }
        if (ce != cudaSuccess) return SSSP_E_CUDA;
        if (cudaMemcpyAsync(&hc, L.ctrl, sizeof(Ctrl), cudaMemcpyDeviceToHost, stream) != cudaSuccess ||
            cudaStreamSynchronize(stream) != cudaSuccess)
            return SSSP_E_CUDA;
        if (hc.error != kErrWide) break;
        // the front is too wide for one cluster: start over on the whole grid
        wg.wide = true;
        cudaMemsetAsync(L.ctrl, 0, sizeof(Ctrl), stream);
    }
    if (hc.error == kErrNone && hc.finished) return SSSP_OK;
    if (hc.error == kErrTimeout) return SSSP_E_TIMEOUT;
    return SSSP_E_CUDA;
}
