// How random runs (mc_walk.cuh) are given to warps and lanes.  Internal.
#pragma once

#include <cstdint>

#include "mc.h"

namespace mc {

// Runs from which each takes a lane (swarm_runs) instead of a warp
// (warp_walk_time).  A warp's 32 lanes share a run's draws (FREE) or its units
// (GREEDY), which is faster while warps wait for work: 4,096 GREEDY runs of
// 64-bit clocks take 58 us a warp each and 70 a lane each, 8,192 82 and 71;
// 32,768 FREE runs of up to 400 work-groups 82 and 106, 131,072 218 and 205.
// (16,384 runs of C1, GREEDY: 45 and 23 us; 1,048,576: 1,262 and 49, and 949
// when a thread took a run step by step.)
constexpr uint32_t kLaneRunsGreedy = 8192;
constexpr uint32_t kLaneRunsFree = 131072;
__host__ __device__ inline uint32_t lane_runs(uint32_t rule) { return rule == MC_GREEDY ? kLaneRunsGreedy : kLaneRunsFree; }
// A run of many models launches the lanes' kernel too when its models may
// together have that many.
inline bool sim_lanes_launch(uint64_t models, uint64_t walks) { return models * walks >= kLaneRunsGreedy; }

}  // namespace mc
