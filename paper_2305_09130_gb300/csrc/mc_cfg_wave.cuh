// Wave units: the configurations of GREEDY models, one warp each (included
// by mc_cfg.cu only).
//
// Under GREEDY only the units with the smallest clock may take the next
// work-group (Listing 5).  Let E be the units whose clock is the smallest,
// m, in some state of a configuration from which every unit of E still has
// to start: taking a work-group moves a unit's clock above m, so the next
// |E| transitions each take another unit of E, in every order, and all orders
// end in the one state in which every unit of E has started.  Call this a
// wave.  From the configuration's select state (all clocks 0) the search is
// a chain of waves, and every state of one level has the form
//     base counts + one work-group for each unit of a subset S of E,
// with the base and E common to the level.  So a level is a set of subsets:
// here a bitmap with one bit per subset, which is the frontier and the
// level's exact visited set at once.  Expanding every state of the level by
// unit q is (level & subsets without q) shifted by 2^q, and two states that
// reach the same successor set the same bit.  Pruning acts on units (the
// successor's time is the starting unit's new clock, all others being within
// the bound already): a unit whose next clock passes T starts in no state, so
// the wave ends early and the search with it.
//
// The chain can be entered at any wave: before instant m unit c has started
// ceil(m / t_c) times (each of its starts is a multiple of t_c), and that state
// was reached if none of those starts ended beyond T.  So a configuration's
// levels can be split into segments explored at the same time; the wave on a
// border is explored on both sides, and each side counts its own levels.
//
// Positions in the bitmap: the units of E in descending index, so the order
// of the bitmap's indices is the order of the packed keys and the smallest
// key is the lowest bit.  Bits 0-4 of an index pick the bit of a lane's word,
// the bits above pick the lane.
//
// What bounds it: the chain of levels of the deepest configuration, a few
// shifts and shuffles each; no memory is read in the loop.  One warp, because
// a level of 2^10 subsets is one word per lane and a wider group would add a
// barrier to every level.  Measured on GB300, counting C3 literal (10 x 6
// configurations of up to 4,096 work-groups, 8 units of one speed, 128-bit
// keys): the pass 4,550 us with block units (a hashed table in shared memory
// and a block barrier per level), 324 us with a warp per configuration, about
// 50 us with a warp per segment; C2 literal's pass (4 units of uneven speeds,
// 1,024 work-groups, almost every wave one unit) 422, 94 and 33 us.  Left: a
// launch's fixed costs, and 31 instructions per level at 5 cycles each, one
// warp to a scheduler.
#pragma once
#include <cstdint>

#include "mc_cfg_wave.h"
#include "mc_device.cuh"

namespace mc {
namespace {

using namespace mc::dev;

__device__ __forceinline__ uint32_t lanes_min(uint32_t v) { return __reduce_min_sync(0xffffffffu, v); }
__device__ __forceinline__ uint64_t lanes_min(uint64_t v) { return warp_min_u64(v); }
__device__ __forceinline__ uint32_t lanes_max(uint32_t v) { return __reduce_max_sync(0xffffffffu, v); }
__device__ __forceinline__ uint64_t lanes_max(uint64_t v) { return ~warp_min_u64(~v); }

// Subsets of a word that lack position q (q < 5).
__device__ __forceinline__ constexpr uint32_t without(int q) {
  return q == 0 ? 0x55555555u : q == 1 ? 0x33333333u : q == 2 ? 0x0F0F0F0Fu : q == 3 ? 0x00FF00FFu : 0x0000FFFFu;
}

// The level after `cur` when the units at the positions of A may start; up[h]
// is all ones where lane bit h is set and position 5 + h is in A.
template <int H>
__device__ __forceinline__ uint32_t wave_step(uint32_t cur, const uint32_t (&keep)[5], const uint32_t (&up)[5]) {
  uint32_t o[H ? H : 1];
#pragma unroll
  for (int h = 0; h < H; ++h) o[h] = __shfl_xor_sync(0xffffffffu, cur, 1 << h);
  uint32_t nxt = (((cur & keep[0]) << 1) | ((cur & keep[1]) << 2)) | (((cur & keep[2]) << 4) | ((cur & keep[3]) << 8)) |
                 ((cur & keep[4]) << 16);
#pragma unroll
  for (int h = 0; h < H; ++h) nxt |= o[h] & up[h];
  return nxt;
}

// A whole wave: e units start in every order (e levels), from the empty
// subset to the full one.  The loop is unrolled, so the masks are constants
// and there is no branch; a level is one step, 53 cycles measured at e = 8
// (three shuffles and a chain of shifts), and its width is counted beside
// it: ten bits per level (at most C(10, 5) states), three levels to a word,
// one sum across the lanes per word instead of one per level (47 cycles
// each).  Lane x < e returns the width of the wave's level x + 1.
template <int e>
__device__ __forceinline__ uint32_t wave_full(uint32_t lane) {
  constexpr int H = e > 5 ? e - 5 : 0;
  uint32_t keep[5], up[5];
#pragma unroll
  for (int q = 0; q < 5; ++q) {
    keep[q] = q < e ? without(q) : 0u;
    up[q] = q < H && ((lane >> q) & 1u) ? 0xFFFFFFFFu : 0u;
  }
  uint32_t cur = H == 0 || lane == 0 ? 1u : 0u;  // (in one word: kept alike in every lane)
  uint32_t w[(e + 2) / 3];
#pragma unroll
  for (int x = 0; x < e; ++x) {
    cur = wave_step<H>(cur, keep, up);
    w[x / 3] = (x % 3 ? w[x / 3] : 0u) + (__popc(cur) << (10 * (x % 3)));
  }
  uint32_t mine = 0;
#pragma unroll
  for (int k = 0; k < (e + 2) / 3; ++k) {
    if (H) w[k] = __reduce_add_sync(0xffffffffu, w[k]);
    mine = lane / 3 == k ? w[k] : mine;
  }
  return (mine >> (10 * (lane % 3))) & 1023u;
}

// The first m levels of a wave in which only the units at the positions of A
// may start (pruning, or the work-groups run out): returns the last level's
// subsets.  The levels are not empty: a subset smaller than A leaves a unit
// to start.  Rare (a configuration's last wave), so not specialised.
// Levels from .. to - 1 of them are counted.
__device__ __forceinline__ uint32_t wave_part(uint32_t A, uint32_t m, uint32_t lane, unsigned long long* level,
                                              uint32_t from, uint32_t to) {
  uint32_t keep[5], up[5];
#pragma unroll
  for (int q = 0; q < 5; ++q) {
    keep[q] = (A >> q) & 1u ? without(q) : 0u;
    up[q] = (A >> (5 + q)) & (lane >> q) & 1u ? 0xFFFFFFFFu : 0u;
  }
  uint32_t cur = lane == 0 ? 1u : 0u;
#pragma unroll 1
  for (uint32_t x = 0; x < m; ++x) {
    cur = A >> 5 ? wave_step<5>(cur, keep, up) : wave_step<0>(cur, keep, up);
    const uint32_t w = __reduce_add_sync(0xffffffffu, __popc(cur));
    if (lane == 0 && x >= from && x < to) atomicAdd(level + 2 * x, (unsigned long long)w);
  }
  return cur;
}

// The subsets of `cur` that hold only positions of A.
__device__ __forceinline__ uint32_t wave_within(uint32_t cur, uint32_t A, uint32_t lane) {
  uint32_t w = (lane & ~(A >> 5)) ? 0u : cur;
#pragma unroll
  for (int q = 0; q < 5; ++q)
    if (!((A >> q) & 1u)) w &= without(q);
  return w;
}

// The clocks of a configuration's units.  Two units: every lane keeps both
// (a wave's start needs no exchange between lanes: 36 cycles against 52).
// More: one unit per lane.
template <class C, int PT>
struct WaveClocks {
  C clk[PT], t[PT];
  __device__ void load(const Params& p, uint32_t cfg, uint32_t) {
#pragma unroll
    for (int c = 0; c < PT; ++c) {
      const bool unit = c < (int)p.P;
      t[c] = unit ? (C)((uint64_t)__ldg(p.cost + cfg) * __ldg(p.speed + c)) : (C)0;
      clk[c] = unit ? (C)0 : (C)~(C)0;  // never the smallest
    }
  }
  // The state before the wave in which the work-group after the first `k`
  // starts (its instant by bisection: the smallest with more than k starts at
  // or before it); returns the work-groups taken by then.
  __device__ uint32_t enter(const Params& p, uint32_t k) {
    C t_min = t[0];
    for (int c = 1; c < PT; ++c) t_min = c < (int)p.P && t[c] < t_min ? t[c] : t_min;
    C lo = 0, hi = (C)k * t_min;
    while (lo < hi) {
      const C mid = lo + (hi - lo) / 2;
      uint64_t starts = 0;
      for (int c = 0; c < PT; ++c) starts += c < (int)p.P ? (uint64_t)(mid / t[c]) + 1 : 0ull;
      if (starts > k) hi = mid;
      else lo = mid + 1;
    }
    uint32_t before = 0;
    for (int c = 0; c < PT; ++c) {
      if (c >= (int)p.P) continue;
      const C n = lo / t[c] + (lo % t[c] ? 1 : 0);
      clk[c] = n * t[c];
      before += (uint32_t)n;
    }
    return before;
  }
  // E: the units whose clock is the smallest; late: those of them whose next
  // clock passes `bound`
  __device__ __forceinline__ void first(C bound, uint32_t& E, uint32_t& late) const {
    C mn = clk[0];
#pragma unroll
    for (int c = 1; c < PT; ++c) mn = clk[c] < mn ? clk[c] : mn;
    E = late = 0;
#pragma unroll
    for (int c = 0; c < PT; ++c) {
      const bool in = clk[c] == mn;
      E |= in ? 1u << c : 0u;
      late |= in && (C)(clk[c] + t[c]) > bound ? 1u << c : 0u;
    }
  }
  __device__ __forceinline__ void advance() {  // the units of E start
    C mn = clk[0];
#pragma unroll
    for (int c = 1; c < PT; ++c) mn = clk[c] < mn ? clk[c] : mn;
#pragma unroll
    for (int c = 0; c < PT; ++c) clk[c] += clk[c] == mn ? t[c] : (C)0;
  }
  // the units of E whose next clock is at most `bound`
  __device__ uint32_t within(uint32_t E, C bound) const {
    uint32_t m = 0;
#pragma unroll
    for (int c = 0; c < PT; ++c) m |= ((E >> c) & 1u) && (C)(clk[c] + t[c]) <= bound ? 1u << c : 0u;
    return m;
  }
  __device__ C largest(uint32_t P) const {
    C mx = 0;
#pragma unroll
    for (int c = 0; c < PT; ++c) mx = c < (int)P && clk[c] > mx ? clk[c] : mx;
    return mx;
  }
  __device__ C next(uint32_t u) const {
    C v = 0;
#pragma unroll
    for (int c = 0; c < PT; ++c) v = c == (int)u ? clk[c] + t[c] : v;
    return v;
  }
  __device__ uint32_t taken(uint32_t u) const {
    uint32_t v = 0;
#pragma unroll
    for (int c = 0; c < PT; ++c) v = c == (int)u ? (uint32_t)(clk[c] / t[c]) : v;
    return v;
  }
};

template <class C>
struct WaveClocks<C, 0> {
  C clk, t, nxt;
  bool unit, in;
  __device__ void load(const Params& p, uint32_t cfg, uint32_t lane) {
    unit = lane < p.P;
    t = unit ? (C)((uint64_t)__ldg(p.cost + cfg) * __ldg(p.speed + lane)) : (C)1;
    clk = unit ? (C)0 : (C)~(C)0;
    nxt = clk + t;
  }
  __device__ uint32_t enter(const Params&, uint32_t k) {
    const C t_min = lanes_min(unit ? t : (C)~(C)0);
    C lo = 0, hi = (C)k * t_min;
    while (lo < hi) {
      const C mid = lo + (hi - lo) / 2;
      // (a unit's starts are capped, so that 32 bits hold the sum)
      const C q = mid / t;
      const uint32_t starts = __reduce_add_sync(0xffffffffu, !unit ? 0u : (uint32_t)(q < (C)k ? q : (C)k) + 1);
      if (starts > k) hi = mid;
      else lo = mid + 1;
    }
    const C n = unit ? lo / t + (lo % t ? 1 : 0) : (C)0;
    if (unit) clk = n * t;
    nxt = clk + t;
    return __reduce_add_sync(0xffffffffu, (uint32_t)n);
  }
  __device__ __forceinline__ void first(C bound, uint32_t& E, uint32_t& late) {
    const C mn = lanes_min(clk);  // (every lane takes part)
    in = unit && clk == mn;
    E = __ballot_sync(0xffffffffu, in);
    late = __ballot_sync(0xffffffffu, in && nxt > bound);
  }
  __device__ __forceinline__ void advance() {
    clk = in ? nxt : clk;
    nxt = clk + t;
  }
  __device__ uint32_t within(uint32_t E, C bound) const {
    return E & __ballot_sync(0xffffffffu, unit && nxt <= bound);
  }
  __device__ C largest(uint32_t) const { return lanes_max(unit ? clk : (C)0); }
  __device__ C next(uint32_t u) const { return __shfl_sync(0xffffffffu, nxt, u); }
  __device__ uint32_t taken(uint32_t u) const { return __shfl_sync(0xffffffffu, (uint32_t)(clk / t), u); }
};

// The positions (see above) of the units `mask`, a subset of E.
__device__ __forceinline__ uint32_t wave_positions(uint32_t E, uint32_t mask, uint32_t lane) {
  return __reduce_or_sync(0xffffffffu, (mask >> lane) & 1u ? 1u << (__popc(E >> lane) - 1) : 0u);
}

// Explore work-groups k0 + 1 .. k1 of configuration `cfg` of pass Q at
// threshold T with one warp (the whole configuration: 0 .. N): the same
// widths, record and early exit as explore_unit.
template <class K, class C, int PT>
__device__ void explore_unit_wave(const CfgPass& Q, uint32_t cfg, uint64_t T, uint32_t k0, uint32_t k1) {
  const uint32_t lane = threadIdx.x & 31u;
  const uint32_t P = Q.p.P, b = Q.p.b;
  const uint32_t i = cfg / b, j = cfg % b;
  const bool early = Q.early_exit != 0;
  const uint32_t N = __ldg(Q.p.N + cfg);
  WaveClocks<C, PT> clocks;
  clocks.load(Q.p, cfg, lane);
  // what pruning compares with: T, saturated at the clock type's maximum
  const C Tc = Q.prune && T < (uint64_t)(C)~(C)0 ? (C)T : (C)~(C)0;
  unsigned long long* const levels = reinterpret_cast<unsigned long long*>(Q.levels);
  Ctrl* const ctrl = Q.ctrl;

  // work-groups taken before the current wave; the first wave's may have
  // started before the segment
  uint32_t sum = k0 ? clocks.enter(Q.p, k0) : 0u;
  const bool reached = k0 == 0 || clocks.largest(P) <= Tc;
  uint32_t E = 0, cur = 0;       // the wave's units, the current level's subsets
  uint32_t ones = 0;             // one-state levels of the current 32-level window
  uint32_t window = (3 + sum) >> 5;
  bool done = false;             // the terminal level was reached
  // early exit: the least level known to hold a violating terminal, asked
  // for at the end of a window and used at the next, so the load never holds
  // a level up (a later stop only explores levels that are not counted).
  // Other units lower the word meanwhile, and it decides which collectives
  // the warp reaches: lane 0 reads it, and all lanes use its value.
  uint32_t asked = 0;  // (lane 0's)
  if (early && lane == 0) asked = ld_relaxed_u32(&ctrl->stop_c);
  bool beyond = false;  // a segment below the first violating level: not counted
  if (k0) {
    const uint32_t cut = __shfl_sync(0xffffffffu, asked, 0);
    beyond = cut && ~cut <= 2 + k0;
  }
  while (reached && !beyond && sum < k1) {
    uint32_t late = 0;
    // waves of one unit, the common ones of uneven speeds: one state per
    // level, one branch per wave; their widths are added window by window
    for (;;) {
      clocks.first(Tc, E, late);
      const uint32_t at = 3 + sum;  // the wave's first level
      if ((E & (E - 1)) | late | (uint32_t)(sum + 1 >= k1) | (uint32_t)((at >> 5) != window)) break;
      ones |= 1u << (at & 31u);
      ++sum;
      clocks.advance();
    }
    const uint32_t before = 2 + sum;  // the level the wave starts from
    if (((before + 1) >> 5) != window) {
      if ((ones >> lane) & 1u) atomicAdd(levels + 2ull * (window * 32 + lane), 1ull);
      ones = 0;
      window = (before + 1) >> 5;
      if (early) {
        const uint32_t known = __shfl_sync(0xffffffffu, asked, 0);
        if (known && ~known <= before) break;  // deeper widths are not counted
        if (lane == 0) asked = ld_relaxed_u32(&ctrl->stop_c);
      }
    }
    const uint32_t e = __popc(E);
    if (late == 0 && sum + e < N) {  // every unit of E starts
      uint32_t width = 1;
      switch (e) {
        case 1: break;
        case 2: width = wave_full<2>(lane); break;
        case 3: width = wave_full<3>(lane); break;
        case 4: width = wave_full<4>(lane); break;
        case 5: width = wave_full<5>(lane); break;
        case 6: width = wave_full<6>(lane); break;
        case 7: width = wave_full<7>(lane); break;
        case 8: width = wave_full<8>(lane); break;
        case 9: width = wave_full<9>(lane); break;
        default: width = wave_full<10>(lane); break;
      }
      // (a wave on the segment's border: its own levels only)
      if (lane < e && sum + lane >= k0 && sum + lane < k1)
        atomicAdd(levels + 2ull * (before + 1 + lane), (unsigned long long)width);
      sum += e;
      clocks.advance();
    } else {  // the last wave: the work-groups run out, or pruning keeps a unit from starting
      const uint32_t A = wave_positions(E, E & ~late, lane);
      const uint32_t m = min(N - sum, (uint32_t)__popc(A));
      cur = wave_part(A, m, lane, levels + 2ull * (before + 1), k0 > sum ? k0 - sum : 0u, k1 - sum);
      sum += m;
      done = sum == N;
      break;
    }
  }
  if ((ones >> lane) & 1u) atomicAdd(levels + 2ull * (window * 32 + lane), 1ull);

  // the terminals (all at level 2 + N): the least time within T, and the
  // smallest key of that time.  A subset's time is the largest clock of the
  // base and of its own units after their start, so the candidates are the
  // units' next clocks, each reached if a subset without later ones exists.
  C tv = (C)~(C)0;
  bool hit = false;
  K key = 0;
  if (done) {
    const C base_mx = clocks.largest(P);
    for (uint32_t rest = E; rest; rest &= rest - 1) {
      const C f = clocks.next(__ffs(rest) - 1);
      const C v = f > base_mx ? f : base_mx;
      if (hit && v >= tv) continue;  // (units of one speed: the same time)
      if (__any_sync(0xffffffffu, wave_within(cur, wave_positions(E, clocks.within(E, v), lane), lane) != 0)) {
        hit = true;
        tv = v;
      }
    }
    hit = hit && (uint64_t)tv <= T;
    if (hit) {
      const uint32_t word = wave_within(cur, wave_positions(E, clocks.within(E, tv), lane), lane);
      const uint32_t who = __ffs(__ballot_sync(0xffffffffu, word != 0)) - 1;
      const uint32_t S = (who << 5) | (uint32_t)(__ffs(__shfl_sync(0xffffffffu, word, who)) - 1);
      key = ((K)(i + 1) << Q.p.wg_shift) | ((K)(j + 1) << Q.p.ts_shift);
      for (uint32_t u = 0; u < P; ++u) {
        const uint32_t in = ((E >> u) & 1u) && ((S >> (__popc(E >> u) - 1)) & 1u) ? 1u : 0u;
        key |= (K)(clocks.taken(u) + in) << ((P - 1 - u) * Q.p.n_bits);
      }
    }
  }
  // the deepest level reached: in the record, and by segments, which share one,
  // in pad1[0] (one word for the pass: taken by every unit of 62,500
  // configurations it lengthened a pass from 425 to 468 us)
  const bool whole = k0 == 0 && k1 == N;
  if (lane == 0 && reached && !whole) atomicMax(&ctrl->pad1[0], 2 + min(sum, k1));
  if (lane == 0 && k1 == N) {
    if (hit && early) atomicMax(&ctrl->stop_c, ~(2u + N));
    CfgRec rec;
    rec.vpack = hit ? pack_tij((uint64_t)tv, i, j) : kNone;
    rec.wkey_lo = hit ? KeyOps<K>::lo(key) : kNone;
    rec.wkey_hi = hit ? KeyOps<K>::hi(key) : kNone;
    rec.widx = 0;  // no log: wave_trace gives the path
    rec.deepest = whole ? 2 + sum : 0u;
    Q.rec[cfg] = rec;
  }
}

// Segment number `part` of a configuration (`segment` work-groups each, 0: the
// whole configuration).
template <class K, class C>
__device__ __forceinline__ void explore_wave(const CfgPass& Q, uint32_t cfg, uint64_t T, uint32_t segment, uint32_t part) {
  const uint32_t N = __ldg(Q.p.N + cfg), k0 = segment * part;
  const uint32_t k1 = segment && N - k0 > segment ? k0 + segment : N;
  if (Q.p.P <= 2) explore_unit_wave<K, C, 2>(Q, cfg, T, k0, k1);
  else explore_unit_wave<K, C, 0>(Q, cfg, T, k0, k1);
}

// The trace s0 -> the witness of configuration (i, j), replayed by one warp:
// wave after wave, the units that the witness's counts say start in it, in
// index order.  Every step takes a unit of the smallest clock, and no clock
// passes the witness's time, so each state on the way was explored.
template <class K>
__device__ void wave_trace(const CfgPass& Q, uint32_t i, uint32_t j, K key) {
  const uint32_t lane = threadIdx.x & 31u;
  const Params& p = Q.p;
  const uint32_t P = p.P, cfg = i * p.b + j;
  const uint32_t N = __ldg(p.N + cfg);
  const bool unit_ok = lane < P;
  const uint64_t t_c = unit_ok ? (uint64_t)__ldg(p.cost + cfg) * __ldg(p.speed + lane) : 0;
  const uint32_t goal = unit_ok ? field(key, (P - 1 - lane) * p.n_bits, p.n_mask) : 0;
  auto put = [&](uint32_t l, K k) {
    Q.trace[2 * l] = KeyOps<K>::lo(k);
    Q.trace[2 * l + 1] = KeyOps<K>::hi(k);
  };
  const K k1 = (K)(i + 1) << p.wg_shift;
  K base = k1 | ((K)(j + 1) << p.ts_shift);
  if (lane < 3) put(lane, lane == 0 ? (K)0 : lane == 1 ? k1 : base);
  uint64_t clk = 0;
  uint32_t n = 0, sum = 0;
  while (sum < N) {
    const uint64_t mn = warp_min_u64(unit_ok ? clk : kNone);
    const bool starts = unit_ok && clk == mn && n < goal;
    const uint32_t S = __ballot_sync(0xffffffffu, starts);
    if (!S) {  // cannot happen: the witness is reached by these steps
      if (lane == 0) set_error(Q.ctrl, MC_ERR_FRONTIER);
      return;
    }
    K k = base;  // after this lane's unit has started
    for (uint32_t u = 0; u < P; ++u) {
      if (!((S >> u) & 1u)) continue;
      const K one = (K)1 << ((P - 1 - u) * p.n_bits);
      base += one;
      if (u <= lane) k += one;
    }
    if (starts) {
      put(2 + sum + __popc(S & ((2u << lane) - 1u)), k);
      clk += t_c;
      ++n;
    }
    sum += __popc(S);
  }
}

}  // namespace
}  // namespace mc
