// fan.h -- host-side declarations of the multi-source kernel (fan.cuh).
#pragma once

#include "fan.cuh"

namespace sssp {

// Launches one group of up to 32 queries cooperatively.
cudaError_t launch_fan(int wt, const FanParams& p, int grid, cudaStream_t stream);
// The first nq columns of rows [n][32] as the caller's [nq][n].
cudaError_t launch_fan_out(const uint32_t* rows, int32_t n, int32_t nq, uint32_t* out, int sms, cudaStream_t stream);

}  // namespace sssp
