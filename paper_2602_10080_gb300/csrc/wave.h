// wave.h -- host-side declarations of the cluster wavefront kernel (wave.cuh).
#pragma once

#include "wave.cuh"

namespace sssp {

// Launches one cluster of 1 << p.log_g blocks per query.
cudaError_t launch_wave(int wt, int pred, const WaveParams& p, int nq, int threads, size_t smem,
                        cudaStream_t stream);
// Launches the whole-grid kernel cooperatively (one query).
cudaError_t launch_tide(int wt, int pred, const WaveParams& p, int grid, int threads, cudaStream_t stream);

}  // namespace sssp
