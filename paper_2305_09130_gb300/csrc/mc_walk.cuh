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
#include "mc_walk.h"

namespace mc {
namespace dev {

// x % d for a divisor below 2^16 that stays the same: d's reciprocal (floor of
// (2^32 - 1) / d) is multiplied instead of a 64-bit division's hundred
// instructions (262,144 runs of C3 literal drew their configurations in three
// quarters of the swarm's time).  A word's quotient comes out exact or one
// short, which one conditional subtraction mends.
struct FastMod {
  uint32_t d, inv, two32;  // two32 = 2^32 % d
  __device__ explicit FastMod(uint32_t x) : d(x), inv(0xFFFFFFFFu / x) {
    const uint32_t rest = 0xFFFFFFFFu - inv * x + 1;
    two32 = rest == x ? 0u : rest;
  }
  __device__ __forceinline__ uint32_t word(uint32_t x) const {
    const uint32_t r = x - __umulhi(x, inv) * d;
    return r >= d ? r - d : r;
  }
  __device__ __forceinline__ uint32_t of(uint64_t x) const {
    return word(word((uint32_t)(x >> 32)) * two32 + word((uint32_t)x));
  }
};

// Of the units `from` (bits, index order), the `left` ones that draws number
// ctr, ctr + 1, ... pick one after another.
__device__ __forceinline__ uint32_t pick_units(uint32_t from, uint32_t left, uint64_t seed, uint64_t ctr) {
  uint32_t picked = 0;
  for (uint32_t x = 0; x < left; ++x) {
    uint32_t b = from;
    for (uint32_t r = FastMod(__popc(from)).of(splitmix64_at(seed, ctr + x)); r; --r) b &= b - 1;
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

// Clocks of a run's units in one thread, PT >= P of them in registers, and the
// division of a 32-bit instant by a unit's time through its reciprocal.
template <class C, int PT>
struct RunUnits {
  C t[PT], clk[PT];
  uint32_t inv[PT];
  __device__ __forceinline__ void load(const Params& p, uint64_t cost) {
#pragma unroll
    for (int c = 0; c < PT; ++c) {
      t[c] = c < (int)p.P ? (C)(cost * __ldg(p.speed + c)) : (C)1;
      clk[c] = 0;
      if (sizeof(C) == 4) inv[c] = 0xFFFFFFFFu / (uint32_t)t[c];
    }
  }
  __device__ __forceinline__ C over(C x, int c) const {  // x / t[c]
    if (sizeof(C) == 8) return x / t[c];
    const uint32_t q = __umulhi((uint32_t)x, inv[c]);  // exact or one short
    return q + ((uint32_t)x - q * (uint32_t)t[c] >= (uint32_t)t[c] ? 1u : 0u);
  }
  __device__ __forceinline__ C largest(uint32_t P) const {
    C mx = 0;
#pragma unroll
    for (int c = 0; c < PT; ++c) mx = c < (int)P && clk[c] > mx ? clk[c] : mx;
    return mx;
  }
};

// Terminal time of a GREEDY run of N work-groups, by one thread: the last
// group's instant by bisection, as warp_walk_time.  `ctr` is the draw of the
// first work-group.
template <class C, int PT>
__device__ __forceinline__ C greedy_run(RunUnits<C, PT>& u, uint32_t P, uint32_t N, uint64_t seed, uint64_t ctr) {
  C t_min = u.t[0];
#pragma unroll
  for (int c = 1; c < PT; ++c) t_min = c < (int)P && u.t[c] < t_min ? u.t[c] : t_min;
  C lo = 0, hi = (C)(N - 1) * t_min;
  while (lo < hi) {
    const C mid = lo + (hi - lo) / 2;
    uint64_t starts = 0;  // at or before mid
#pragma unroll
    for (int c = 0; c < PT; ++c) starts += c < (int)P ? (uint64_t)u.over(mid, c) + 1 : 0ull;
    if (starts >= N) hi = mid;
    else lo = mid + 1;
  }
  uint32_t before = 0, E = 0;
#pragma unroll
  for (int c = 0; c < PT; ++c) {
    if (c >= (int)P) continue;
    const C q = u.over(lo, c);
    const bool in = q * u.t[c] == lo;
    E |= in ? 1u << c : 0u;
    const C n = in ? q : q + 1;  // starts before the instant
    before += (uint32_t)n;
    u.clk[c] = n * u.t[c];
  }
  const uint32_t left = N - before;
  const uint32_t S = left < (uint32_t)__popc(E) ? pick_units(E, left, seed, ctr + before) : E;
#pragma unroll
  for (int c = 0; c < PT; ++c) u.clk[c] += (S >> c) & 1u ? u.t[c] : (C)0;
  return u.largest(P);
}

// Runs first .. last - 1 (numbered from w0) by one warp: this lane's least
// (time << 24 | run) over those that end at or below `bound`, kNone if none
// does.  Clocks in C, PT >= P of them in registers.  GREEDY runs cost the same
// whatever their length; FREE runs are stepped through, and a lane takes the
// warp's next run as soon as its own ends or passes the bound, so that lanes
// do not wait for the longest of 32.  262,144 runs of C3 literal: 13.2 ms by
// single steps with the clocks in local memory, 0.38 ms group by group (the
// longest run's 512 groups in a row); the search of two rounds takes 0.11 ms
// here, most of it launches and waits.
template <class C, int PT>
__device__ unsigned long long swarm_runs(const Params& p, uint64_t seed, uint64_t w0, uint32_t first, uint32_t last,
                                         uint64_t bound) {
  const uint32_t lane = threadIdx.x & 31u;
  unsigned long long best = kNone;
  const C cut = bound < (uint64_t)(C)~(C)0 ? (C)bound : (C)~(C)0;
  const FastMod mod_a(p.a), mod_b(p.b), mod_P(p.P);
  RunUnits<C, PT> u;
  uint32_t N = 0, sum = 0, k = 0;
  uint64_t ctr = 0;
  auto start = [&]() {
    ctr = (w0 + k) << 32;
    const uint32_t i = mod_a.of(splitmix64_at(seed, ctr)), j = mod_b.of(splitmix64_at(seed, ctr + 1));
    const uint32_t cfg = i * p.b + j;
    N = __ldg(p.N + cfg);
    u.load(p, __ldg(p.cost + cfg));
    sum = 0;
  };
  auto finish = [&](C time) {
    if (time > cut) return;
    const unsigned long long v = ((unsigned long long)time << 24) | k;
    best = v < best ? v : best;
  };
  if (p.rule == MC_GREEDY) {
    for (k = first + lane; k < last; k += 32) {
      start();
      finish(greedy_run<C, PT>(u, p.P, N, seed, ctr + 2));
    }
    return best;
  }
  bool running = false;
  for (uint32_t next = first;;) {  // (uniform)
    const uint32_t idle = __ballot_sync(0xffffffffu, !running);
    if (idle == 0xFFFFFFFFu && next >= last) break;
    k = running ? k : next + __popc(idle & ((1u << lane) - 1u));
    next += __popc(idle);
    if (!running && k < last) {
      start();
      running = true;
    }
    if (!running) continue;
    const uint32_t c0 = mod_P.of(splitmix64_at(seed, ctr + 2 + sum));
    C at = 0;
#pragma unroll
    for (int c = 0; c < PT; ++c) {
      u.clk[c] += c == (int)c0 ? u.t[c] : (C)0;
      at = c == (int)c0 ? u.clk[c] : at;
    }
    const bool end = ++sum == N;
    if (end && at <= cut) finish(u.largest(p.P));
    running = !end && at <= cut;  // (a clock beyond the bound: the run cannot end within it)
  }
  return best;
}

}  // namespace dev
}  // namespace mc
