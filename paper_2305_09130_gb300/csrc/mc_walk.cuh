// Terminal times of random runs (Section 4, Step 3: T_ini; Section 5: the
// swarm).  Run w draws splitmix64 outputs number (w << 32) + 0, 1, ...: the WG
// index, the TS index, then per work-group the unit among the allowed ones in
// index order (walk_time in mc_device.cuh steps through one).  These give the
// same times without every step:
//
//   GREEDY  the units with the smallest clock all start before any other
//           clock is the smallest again (each start raises one of them), in
//           whatever order the draws pick them, so the draws only matter in
//           the last such group, where the work-groups run out.  The clocks
//           before it follow from its instant alone;
//   FREE    a clock is the number of draws that picked its unit, so the
//           draws can be taken in any order.
#pragma once
#include <cstdint>

#include "mc_device.cuh"

namespace mc {
namespace dev {

// Of the units `from` (bits, index order), the `left` ones that draws number
// ctr, ctr + 1, ... pick one after another.
__device__ __forceinline__ uint32_t pick_units(uint32_t from, uint32_t left, uint64_t seed, uint64_t ctr) {
  uint32_t picked = 0;
  for (uint32_t x = 0; x < left; ++x) {
    uint32_t b = from;
    for (uint32_t r = (uint32_t)(splitmix64_at(seed, ctr + x) % __popc(from)); r; --r) b &= b - 1;
    b &= 0u - b;
    picked |= b;
    from ^= b;
  }
  return picked;
}

__device__ __forceinline__ uint64_t warp_max_u64(uint64_t v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const uint64_t w = __shfl_xor_sync(0xffffffffu, v, o);
    v = w > v ? w : v;
  }
  return v;
}
__device__ __forceinline__ uint64_t warp_sum16(uint64_t v) {  // over the low 16 lanes, in each of them
#pragma unroll
  for (int o = 8; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Terminal time of run w, by one warp (lane c holds unit c).  GREEDY: the
// last group's instant m is the smallest with sum_c (floor(m / t_c) + 1) >= N
// starts at or before it, found by bisection (at most 40 steps where the run
// has N).  Measured: the simulation of a C2 query (up to 1,024 work-groups)
// 80 us by steps in one thread, 8 us here; of 256 models in a batch, 342 ->
// 12 us.
__device__ inline uint64_t warp_walk_time(const Params& p, uint64_t seed, uint64_t w) {
  const uint32_t lane = threadIdx.x & 31u;
  const uint64_t ctr = w << 32;
  const uint32_t i = (uint32_t)(splitmix64_at(seed, ctr) % p.a);
  const uint32_t j = (uint32_t)(splitmix64_at(seed, ctr + 1) % p.b);
  const uint32_t cfg = i * p.b + j;
  const uint32_t N = __ldg(p.N + cfg);
  const bool unit = lane < p.P;
  const uint64_t t = unit ? (uint64_t)__ldg(p.cost + cfg) * __ldg(p.speed + lane) : 1;
  uint64_t clk = 0;
  if (p.rule == MC_FREE) {
    uint32_t n = 0;
    for (uint32_t k = 0; k < N; k += 32) {
      const uint32_t c = k + lane < N ? (uint32_t)(splitmix64_at(seed, ctr + 2 + k + lane) % p.P) : 32u;
      for (uint32_t u = 0; u < p.P; ++u) {
        const uint32_t m = __ballot_sync(0xffffffffu, c == u);
        if (lane == u) n += __popc(m);
      }
    }
    clk = n * t;
  } else {
    const uint64_t t_min = ~warp_max_u64(unit ? ~t : 0ull);
    uint64_t lo = 0, hi = (uint64_t)(N - 1) * t_min;  // the fastest unit alone starts N by then
    while (lo < hi) {
      const uint64_t mid = lo + (hi - lo) / 2;
      // (a unit's starts are capped at N, so the sum cannot wrap)
      const uint64_t q = (p.clk32 ? (uint32_t)mid / (uint32_t)t : mid / t) + 1;
      if (__shfl_sync(0xffffffffu, warp_sum16(unit ? (q < N ? q : N) : 0ull), 0) >= N) hi = mid;
      else lo = mid + 1;
    }
    const uint64_t n = unit ? (lo + t - 1) / t : 0;  // starts before the instant
    const uint32_t before = (uint32_t)__shfl_sync(0xffffffffu, warp_sum16(n), 0);
    const uint32_t E = __ballot_sync(0xffffffffu, unit && n * t == lo);
    const uint32_t S = pick_units(E, N - before, seed, ctr + 2 + before);
    clk = (n + ((S >> lane) & 1u)) * t;
  }
  return warp_max_u64(unit ? clk : 0ull);
}

// The runs first, first + stride, ... below `walks` (numbered from w0) of one
// thread: the least (time << 24 | run) over those that end at or below
// `bound`, kNone if none does.  A thread takes its next run as soon as one
// ends, so a warp's lanes do not wait for the longest of 32 runs (on C3
// literal runs have 8 to 4,096 work-groups, on average 819).  Clocks in C,
// PT >= P of them in registers.  Bound by instructions: 262,144 runs of C3
// literal 13.2 ms by single steps with the clocks in local memory, 0.40 ms
// here.
template <class C, int PT>
__device__ unsigned long long swarm_runs(const Params& p, uint64_t seed, uint64_t w0, uint64_t first, uint64_t stride,
                                         uint32_t walks, uint64_t bound) {
  unsigned long long best = kNone;
  const C cut = bound < (uint64_t)(C)~(C)0 ? (C)bound : (C)~(C)0;
  C clk[PT], t[PT];
  uint32_t N = 0, sum = 0;
  uint64_t ctr = 0;
  bool running = false;
  for (uint64_t k = first; k < walks;) {
    if (!running) {
      ctr = (w0 + k) << 32;
      const uint32_t i = (uint32_t)(splitmix64_at(seed, ctr) % p.a);
      const uint32_t j = (uint32_t)(splitmix64_at(seed, ctr + 1) % p.b);
      const uint32_t cfg = i * p.b + j;
      N = __ldg(p.N + cfg);
      const uint32_t cost = __ldg(p.cost + cfg);
#pragma unroll
      for (int c = 0; c < PT; ++c) {
        t[c] = c < (int)p.P ? (C)((uint64_t)cost * __ldg(p.speed + c)) : (C)0;
        clk[c] = c < (int)p.P ? (C)0 : (C)~(C)0;
      }
      sum = 0;
      running = true;
    }
    bool end, over = false;
    if (p.rule == MC_GREEDY) {
      C mn = clk[0];
#pragma unroll
      for (int c = 1; c < PT; ++c) mn = clk[c] < mn ? clk[c] : mn;
      uint32_t E = 0;
#pragma unroll
      for (int c = 0; c < PT; ++c) E |= clk[c] == mn ? 1u << c : 0u;
      const uint32_t e = __popc(E);
      end = sum + e >= N;
      over = mn > cut;  // a clock passed the bound: the run cannot end within it
      const uint32_t S = sum + e > N ? pick_units(E, N - sum, seed, ctr + 2 + sum) : E;
      sum += e;
#pragma unroll
      for (int c = 0; c < PT; ++c) clk[c] += (S >> c) & 1u ? t[c] : (C)0;
    } else {
      const uint32_t u = (uint32_t)(splitmix64_at(seed, ctr + 2 + sum) % p.P);
      C at = 0;
#pragma unroll
      for (int c = 0; c < PT; ++c) {
        clk[c] += c == (int)u ? t[c] : (C)0;
        at = c == (int)u ? clk[c] : at;
      }
      over = at > cut;
      end = ++sum == N;
    }
    if (end || over) {
      C mx = 0;
#pragma unroll
      for (int c = 0; c < PT; ++c) mx = c < (int)p.P && clk[c] > mx ? clk[c] : mx;
      if (!over && mx <= cut) {
        const unsigned long long v = ((unsigned long long)mx << 24) | k;
        best = v < best ? v : best;
      }
      k += stride;
      running = false;
    }
  }
  return best;
}

}  // namespace dev
}  // namespace mc
