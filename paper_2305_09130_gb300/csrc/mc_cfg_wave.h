// Wave units of the configuration engine (mc_cfg_wave.cuh): which models
// take them.  Internal.
#pragma once

#include <cstdint>

#include "mc.h"

namespace mc {

// A GREEDY configuration of at most kWaveMaxP units is explored by one warp
// with its level as a bitmap over the subsets of the units that start at the
// current instant: 2^P bits, one 32-bit word per lane, so 2^10 subsets fill
// the warp.  (Above, a level needs several words per lane and the block
// units' hashed tables take over.)  Faster than the block units at every P:
// counts of 60 configurations of 4,096 work-groups, each whole, one speed,
// take 0.24 ms against 3.4 ms (P = 1), 0.46 / 3.6 (2), 0.32 / 3.7 (4),
// 0.34 / 4.6 (8), and of 1,024 work-groups 0.11 / 3.7 ms (10).
// mc_options.unit_threads asks for blocks.
constexpr uint32_t kWaveMaxP = 10;

inline bool wave_model(uint32_t rule, uint32_t P, uint32_t unit_threads) {
  return rule == MC_GREEDY && P <= kWaveMaxP && unit_threads == 0;
}

// Configurations whose passes keep a frontier log: block units of GREEDY
// models.  Wave units and every FREE unit build the trace from the witness's
// counts, so no memory is set aside for them (C3 literal in a batch: 0.27 MB
// instead of 68.9).
inline bool cfg_keeps_log(uint32_t rule, bool warp_units) { return rule == MC_GREEDY && !warp_units; }

// A single model's launch splits a configuration's levels into segments of
// this many work-groups (more when a configuration would have over 255), each
// explored by a warp of its own: the state in which every wave before an
// instant has run is known (see mc_cfg_wave.cuh), so segments need not wait
// for each other.  C3 literal's configurations of 4,096 work-groups are 32
// warps instead of one.  A batch has more warps to begin with and pays for a
// unit on the host too, so its segments are longer (256 models: 1,010 us a run
// with configurations whole, 820 in segments of 512); a job of the request
// loop takes configurations whole (its units are listed while requests wait:
// 48 C3 requests take 1,060 us, and 1,070 in segments).
constexpr uint32_t kWaveSegment = 128;
constexpr uint32_t kWaveRunSegment = 512;

inline uint32_t wave_segment(uint32_t n_max, uint32_t length = kWaveSegment) {
  if (n_max >= 1u << 27) return 0;  // (the search for a segment's start sums starts in 32 bits)
  const uint32_t least = (uint32_t)(((uint64_t)n_max + 254) / 255);
  return least > length ? least : length;
}
inline uint64_t wave_segments(uint32_t n, uint32_t segment) { return ((uint64_t)n + segment - 1) / segment; }

}  // namespace mc
