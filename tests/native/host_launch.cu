// A launch with little shared memory leaves a function's limit where a launch
// with much, by another thread at the same time, needs it.
#include <cstdio>
#include <cstdlib>

#include "api_internal.h"
#include "fake_cuda.h"

using namespace sssp;

static int least_limit() {
    std::lock_guard<std::mutex> lk(fake::mu);
    int least = 1 << 30;
    for (auto& f : fake::max_shared) least = std::min(least, f.second);
    fake::max_shared.clear();
    return least;
}

int main() {
    WaveParams P;
    std::memset(&P, 0, sizeof(P));
    for (int log_g : {0, 4})
        for (int hops : {1, 8})
            for (size_t smem : {(size_t)1024, kWaveMaxShared, (size_t)2048}) {
                P.log_g = log_g;
                P.hops = hops;
                CHECK(launch_wave(0, 1, P, 1, 128, smem, nullptr) == cudaSuccess);
                if (smem == 2048) CHECK(least_limit() >= (int)kWaveMaxShared);
            }
    KernelKey key{0, 0, 0};
    KParams K;
    std::memset(&K, 0, sizeof(K));
    const size_t much = 100 * 1024;
    int blocks = 0;
    launch_mlmq(key, dim3(1), dim3(32), much, nullptr, K);
    launch_mlmq(key, dim3(1), dim3(32), 4096, nullptr, K);
    CHECK(least_limit() >= (int)much);
    occupancy_mlmq(key, 256, much, &blocks);
    occupancy_mlmq(key, 256, 4096, &blocks);
    CHECK(least_limit() >= (int)much);
    // more than the device has stays refused
    CHECK(launch_mlmq(key, dim3(1), dim3(32), 228 * 1024, nullptr, K) != cudaSuccess);
    std::puts("ok");
    return 0;
}
