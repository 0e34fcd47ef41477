// wave.h -- host-side declarations of the cluster wavefront kernel (wave.cuh).
#pragma once

#include <condition_variable>
#include <cstddef>
#include <mutex>
#include <set>

#include "wave.cuh"

namespace sssp {

// How a call without a configuration is run: one cluster per query (wave),
// the whole grid on one query (tide), the queries one after the other, or 32
// queries side by side (fan).
enum WaveKind { kOneCluster, kWholeGrid, kInTurn, kSideBySide };

struct WavePlan {
    WaveKind kind = kOneCluster;
    int log_g = 0;         // log2 of a cluster's blocks
    int threads = 1024;
    uint32_t front = 1;
    double delta = 1.0;
    int32_t hops = 1;
    int32_t hub_deg = 256;
    uint32_t wide = kInfU32;
    bool core = false;     // tide: leave the core's heavy arcs out (WaveGraph::core)
    int32_t core_deg = 256;
};

// What the plan depends on.  wide: a solve found the front too wide for one
// cluster; deep: a batch side by side took too many steps; steps: the most that
// a single query has taken (0: none yet).
struct WaveGraph {
    int32_t n;
    int64_t m;
    double avg_w, max_deg;
    int sms;
    bool wide;
    // symmetric, hubs, rows with their light arcs first: for a batch side by
    // side, and (few light arcs) for one query
    bool core, core_one;
    bool deep;
    int64_t steps;
};

constexpr int kTideLogWords = 17;               // the grid kernel spreads the places over at least 2^17 words
constexpr size_t kWaveMaxShared = 176 * 1024;   // pending words of one block (beside WaveShared)

// The kernel and launch shape of a call; false: the queue engine takes it.
// A mesh or a road map: few arcs a vertex, and none with many more.
inline bool thin_graph(double deg, double max_deg) {
    return deg <= 6.5 && max_deg <= (2.0 * deg + 1.5 < 11.5 ? 2.0 * deg + 1.5 : 11.5);
}
bool plan_wave(const WaveGraph& g, int32_t nq, int pred_mode, WavePlan* w);
// Steps from which on a batch side by side may give up (see FanParams).
uint32_t deep_steps(int64_t m);
// How many queries on a graph of many steps are taken in turn at most.
int32_t in_turn_limit(const WaveGraph& g);
// The fields of the parameters that follow from the plan; returns the dynamic
// shared memory of a block.
size_t wave_params(const WavePlan& w, const WaveGraph& g, bool f32, bool unit, WaveParams* p);
// The most hub slices of one step: a hub is listed once, in slices of
// kTideChunk arcs.
uint32_t tide_slices(int64_t m, int32_t hub_deg);
// The blocks of a whole-grid kernel wait for one another, so that two of them
// (of two graphs, on two streams) must not share the device half and half: one
// runs at a time, held from the launch to the end of the call, in the order in
// which they asked.  Nobody who has a place or the turn waits for a graph's lock
// or for work that others have queued.
class GridTurns {
public:
    uint64_t take();              // a place in the order
    bool mine(uint64_t place);    // its turn has come
    void wait(uint64_t place);
    void leave(uint64_t place);   // gives up the turn, or the place before it

private:
    std::mutex mu_;
    std::condition_variable cv_;
    uint64_t next_ = 0, now_ = 0;
    std::set<uint64_t> left_;     // places given up before their turn
};
GridTurns& grid_turns(int device);

// A call's turn, until its end.
class GridTurn {
public:
    explicit GridTurn(int device) : turns_(grid_turns(device)) {}
    ~GridTurn() { end(); }
    void wait() {
        place_ = turns_.take();
        has_ = true;
        turns_.wait(place_);
    }
    void end() {
        if (has_) turns_.leave(place_);
        has_ = false;
    }

private:
    GridTurns& turns_;
    uint64_t place_ = 0;
    bool has_ = false;
};

// Launches one cluster of 1 << p.log_g blocks per query.
cudaError_t launch_wave(int wt, int pred, const WaveParams& p, int nq, int threads, size_t smem,
                        cudaStream_t stream);
// Launches the whole-grid kernel cooperatively (one query).
cudaError_t launch_tide(int wt, int pred, const WaveParams& p, int grid, int threads, cudaStream_t stream);

}  // namespace sssp
