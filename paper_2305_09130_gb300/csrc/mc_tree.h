// Ordered expansion of FREE models on the level engine (mc_tree.cu).
// Internal.
#pragma once

#include "mc_internal.h"

namespace mc {

constexpr int kTreeThreads = 256;  // threads per block (mc_options.threads_per_block: fewer)

// 128-bit models whose packed states use at most this many bits are computed
// in 64 bits (stored in 128; the tag of a log entry sits in its low word's
// spare top bits and fills its high word).
constexpr uint32_t kTreeNarrow = 56;

// Bits that tag a log entry with its pass, given the general pass's choice.
inline uint32_t tree_tag_bits(int key_words, uint32_t used_bits, uint32_t tag_bits) {
  const uint32_t room = key_words == 2 && used_bits <= kTreeNarrow ? 64 - used_bits : tag_bits;
  return tag_bits < room ? tag_bits : room;
}

// `used_bits`: bits of a packed state.
int tree_occupancy(int key_words, uint32_t used_bits, int threads, int* blocks_per_sm);
cudaError_t launch_tree(int key_words, uint32_t used_bits, int grid, int threads, const ExploreArgs& args,
                        cudaStream_t stream);

}  // namespace mc
