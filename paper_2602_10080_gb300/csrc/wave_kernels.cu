// wave_kernels.cu -- instantiations of the cluster wavefront kernel and their launch.
#include "internal.h"
#include "wave.h"

namespace sssp {

template <int WT, int PRED, bool CL, int HOPS>
static cudaError_t launch_hops(const WaveParams& p, int nq, int threads, size_t smem, cudaStream_t stream) {
    auto fn = wave_kernel<WT, PRED, CL, HOPS>;
    static std::atomic<int> room[kMaxDevices];
    cudaError_t e = open_shared(fn, smem, room);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t c{};
    c.gridDim = dim3((unsigned)nq << p.log_g);
    c.blockDim = dim3(threads);
    c.dynamicSmemBytes = smem;
    c.stream = stream;
    cudaLaunchAttribute at[1];
    if (CL) {
        if (p.log_g > 3 && (e = cudaFuncSetAttribute(fn, cudaFuncAttributeNonPortableClusterSizeAllowed, 1)) != cudaSuccess)
            return e;
        at[0].id = cudaLaunchAttributeClusterDimension;
        at[0].val.clusterDim.x = 1u << p.log_g;
        at[0].val.clusterDim.y = 1;
        at[0].val.clusterDim.z = 1;
        c.attrs = at;
        c.numAttrs = 1;
    }
    return cudaLaunchKernelEx(&c, fn, p);
}

template <int WT, int PRED, bool CL>
static cudaError_t launch_one(const WaveParams& p, int nq, int threads, size_t smem, cudaStream_t stream) {
    if (p.quads && p.hops > 1) return launch_hops<WT, PRED, CL, kHopsQuads>(p, nq, threads, smem, stream);
    return p.hops > 1 ? launch_hops<WT, PRED, CL, 1>(p, nq, threads, smem, stream)
                      : launch_hops<WT, PRED, CL, 0>(p, nq, threads, smem, stream);
}

template <int WT, int PRED>
static cudaError_t launch_tide_one(const WaveParams& p, int grid, int threads, cudaStream_t stream) {
    cudaLaunchConfig_t c{};
    c.gridDim = dim3(grid);
    c.blockDim = dim3(threads);
    c.stream = stream;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeCooperative;
    at[0].val.cooperative = 1;
    c.attrs = at;
    c.numAttrs = 1;
    if (p.mid || p.pull) return cudaLaunchKernelEx(&c, tide_kernel<WT, PRED, 0, true>, p);
    if (p.quads && p.hops > 1) return cudaLaunchKernelEx(&c, tide_kernel<WT, PRED, kHopsQuads, false>, p);
    return p.hops > 1 ? cudaLaunchKernelEx(&c, tide_kernel<WT, PRED, 1, false>, p)
                      : cudaLaunchKernelEx(&c, tide_kernel<WT, PRED, 0, false>, p);
}

cudaError_t launch_tide(int wt, int pred, const WaveParams& p, int grid, int threads, cudaStream_t stream) {
    if (wt == 0) {
        if (pred == 0) return launch_tide_one<0, 0>(p, grid, threads, stream);
        if (pred == 1) return launch_tide_one<0, 1>(p, grid, threads, stream);
        return launch_tide_one<0, 2>(p, grid, threads, stream);
    }
    return pred == 0 ? launch_tide_one<1, 0>(p, grid, threads, stream)
                     : launch_tide_one<1, 2>(p, grid, threads, stream);
}

template <int WT, int PRED>
static cudaError_t launch_cl(const WaveParams& p, int nq, int threads, size_t smem, cudaStream_t stream) {
    return p.log_g > 0 ? launch_one<WT, PRED, true>(p, nq, threads, smem, stream)
                       : launch_one<WT, PRED, false>(p, nq, threads, smem, stream);
}

cudaError_t launch_wave(int wt, int pred, const WaveParams& p, int nq, int threads, size_t smem,
                        cudaStream_t stream) {
    // fp32 predecessors always follow the strict-improvement rule (2)
    if (wt == 0) {
        if (pred == 0) return launch_cl<0, 0>(p, nq, threads, smem, stream);
        if (pred == 1) return launch_cl<0, 1>(p, nq, threads, smem, stream);
        return launch_cl<0, 2>(p, nq, threads, smem, stream);
    }
    return pred == 0 ? launch_cl<1, 0>(p, nq, threads, smem, stream)
                     : launch_cl<1, 2>(p, nq, threads, smem, stream);
}

}  // namespace sssp
