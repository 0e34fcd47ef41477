// fan.h -- host-side declarations of the multi-source kernel (fan.cuh).
#pragma once

#include <cstddef>

#include "fan.cuh"

namespace sssp {

// Buffers of one group: 4-byte words (barrier, waiting words, rows) and
// 16-byte slices (short rows after them), carved into the parameters.
size_t fan_words(int32_t n, bool pred);
size_t fan_slices(int32_t n, int64_t m);
void fan_carve(uint32_t* words, uint4* slices, int32_t n, int64_t m, bool pred, FanParams* p);
// Launches one group of up to 32 queries cooperatively.
cudaError_t launch_fan(int wt, const FanParams& p, int grid, cudaStream_t stream);
// The first nq columns of rows [n][32] as the caller's [nq][n].
cudaError_t launch_fan_out(const uint32_t* rows, int32_t n, int32_t nq, uint32_t* out, int sms, cudaStream_t stream);

}  // namespace sssp
