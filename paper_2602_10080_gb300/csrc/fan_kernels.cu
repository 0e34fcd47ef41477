// fan_kernels.cu -- instantiations of the multi-source kernel and their launch.
#include <algorithm>

#include "fan.h"

namespace sssp {

template <int WT, bool CORE>
static cudaError_t launch_one(const FanParams& p, int grid, cudaStream_t stream) {
    cudaLaunchConfig_t c{};
    c.gridDim = dim3(grid);
    c.blockDim = dim3(kFanThreads);
    c.stream = stream;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeCooperative;
    at[0].val.cooperative = 1;
    c.attrs = at;
    c.numAttrs = 1;
    return cudaLaunchKernelEx(&c, fan_kernel<WT, CORE>, p);
}

cudaError_t launch_fan(int wt, const FanParams& p, int grid, cudaStream_t stream) {
    if (p.mid) return wt == 0 ? launch_one<0, true>(p, grid, stream) : launch_one<1, true>(p, grid, stream);
    return wt == 0 ? launch_one<0, false>(p, grid, stream) : launch_one<1, false>(p, grid, stream);
}

cudaError_t launch_fan_out(const uint32_t* rows, int32_t n, int32_t nq, uint32_t* out, int sms, cudaStream_t stream) {
    const int tiles = (n + 31) / 32;
    fan_out_kernel<<<std::min(tiles, sms * 8), 256, 0, stream>>>(rows, n, nq, out);
    return cudaGetLastError();
}

}  // namespace sssp
