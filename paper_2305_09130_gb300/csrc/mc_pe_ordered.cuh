// Ordered expansion of the processing-element level model (included by
// mc_pe.cu only): every state is generated once, so no visited set is kept.
//
// Between two clock ticks a unit's events -- taking a work-group, a PE's mark,
// passing a barrier -- depend on that unit alone (and a dispatch on work being
// left, which every order of the same dispatches finds), so events of
// different units commute.  A state is therefore proposed in one order only:
// all events of unit 0 since the last tick first, then unit 1's, and inside a
// unit's step the marks by PE index.  A unit acts only when no later unit has
// acted since the last tick.  By commuting, every state of the general pass
// is reached this way, at the same level and through states of no larger
// time (so pruning keeps them); and the state names its one predecessor: take
// back the last event of the last unit that acted, or the tick when none has.
// Whether unit c has acted since the last tick shows in the state: it is busy
// and its step is marked, or was entered by a dispatch or a barrier; or it is
// idle, its program ends with a barrier, and its clock is the state's time
// (ticks only pass an idle unit by when no work is left, and then leave its
// clock behind).
//
// One thread decodes one state: its successors are a bitmask over the slots
// of propose() (marks, release or dispatch per unit, tick) and their places
// are reserved block by block.  A state just after a tick has up to P*M
// successors and most have one or none, so a warp's successors are then dealt
// evenly to its lanes (a lane finds the state that owns its place by a search
// over the warp's running counts).  The log is tagged where the keys leave room (mc_explore.cuh), so
// a block arrives at the level barrier with its last reservation.
//
// Levels of at most kPeSoloEnter states are explored by block 0 alone, the
// frontier in shared memory and a block barrier per level, until one is wider
// than kPeSoloCap; the other blocks wait at a device-wide barrier, which block
// 0 joins in time for their wait limit (pe_solo_mask).  (Deep programs run
// thousands of levels of a few dozen states.)  What bounds it:
// the chain of a level -- decode, reserve, poll -- not bytes or instructions
// (a fifth of the issue slots are used).  Min-time queries of the abstract
// kernel's model (39M states, 1,531 levels) 57.2 -> 21.0 ms against the pass
// with a visited set, of the Minimum kernel's (3.7M states, 5,141 levels) 29.7
// -> 12.6 ms.
#pragma once
#include <cstdint>

#include "mc_device.cuh"
#include "mc_explore.cuh"

namespace mc {
namespace {

constexpr int kPeThreads = 512;
constexpr int kPeKeys = 2;               // states per thread and tile
constexpr uint32_t kPeSoloCap = 1024;    // states of a level in shared memory
constexpr uint32_t kPeSoloEnter = 512;
constexpr uint32_t kPeSoloLine = 3;      // the barrier's spare line: how block 0's levels ended

// Block 0 leaves the narrow levels at every level that is a multiple of a power
// of two (and the other blocks come back with it), so that their wait stays
// within the wait limit however many narrow levels there are: ten times what
// one takes (2.4 us) for each.  One mask of the level, because the loop is a
// chain that shows every instruction: with the clock read at the levels, or a
// last level kept in a register, searches of the Minimum kernel's model took
// 2 to 3% longer.
constexpr uint64_t kPeSoloLevelNs = 24000;
inline uint32_t pe_solo_mask(uint64_t timeout_ns) {
  uint32_t every = 1;  // (levels stay below 2^30)
  while (every < 1u << 30 && 2ull * every * kPeSoloLevelNs <= timeout_ns) every *= 2;
  return every - 1;
}

struct PeSoloShared {
  u128 keys[2][kPeSoloCap];
};

// What a thread keeps of its state until its successors are written.
struct PeOwn {
  u128 key;
  uint32_t slots;  // successors, by slot
};

// The unit fields of a key, from the last unit (the key's low bits) up.
// SMALL: fields of at most 32 bits, taken by funnel shifts.
template <bool SMALL>
struct PeFields {
  uint32_t w0, w1, w2, w3;
  uint64_t mask;
  uint32_t bits;
  u128 key;
  __device__ PeFields(u128 k, const PeParams& p) : mask(p.unit_mask), bits(p.unit_bits), key(k) {
    if (SMALL) {
      w0 = (uint32_t)k;
      w1 = (uint32_t)(k >> 32);
      w2 = (uint32_t)(k >> 64);
      w3 = (uint32_t)(k >> 96);
    }
  }
  __device__ __forceinline__ uint64_t take() {
    if (!SMALL) {
      const uint64_t f = (uint64_t)key & mask;
      key >>= bits;
      return f;
    }
    const uint32_t f = w0 & (uint32_t)mask;
    w0 = __funnelshift_rc(w0, w1, bits);  // (a shift of 32 moves a whole word)
    w1 = __funnelshift_rc(w1, w2, bits);
    w2 = __funnelshift_rc(w2, w3, bits);
    w3 = bits >= 32 ? 0u : w3 >> bits;
    return f;
  }
};

// Decode `key` and find its successors; a FIN successor within T lowers
// `best`.  PT >= P: units handled without a branch.
template <int PT, bool SMALL>
__device__ __forceinline__ uint32_t pe_slots(const PeParams& p, u128 key, bool prune, uint64_t T, uint64_t& best) {
  using F = typename std::conditional<SMALL, uint32_t, uint64_t>::type;
  const uint32_t i = (uint32_t)((uint64_t)(key >> p.wg_shift) & p.wg_mask) - 1;
  const uint32_t j = (uint32_t)((uint64_t)(key >> p.ts_shift) & p.ts_mask) - 1;
  const uint4 cfg = __ldg(p.cfg4 + i * p.b + j);  // {work-groups, ticks, steps | ends with a barrier, first step}
  const uint32_t S = cfg.z & 0x7FFFFFFFu, pcb = p.pc_bits, M = p.M, P = p.P;
  const uint32_t PM = P * M;
  const F pc_mask = ((F)1 << pcb) - 1;
  PeFields<SMALL> fields(key, p);
  F f[PT];
  uint2 st[PT];
#pragma unroll
  for (int x = 0; x < PT; ++x) {  // x-th field from below: unit P-1-x
    f[x] = x < (int)P ? (F)fields.take() : (F)0;
    const bool busy = (f[x] >> (M + pcb)) & 1u;
    st[x] = busy ? __ldg(p.step + cfg.w + (uint32_t)((f[x] >> M) & pc_mask)) : make_uint2(0, 0);
  }
  uint32_t taken = 0, busy = 0, acted = 0, marks = 0, moves = 0, leaving = 0;
  uint64_t time = 0;
  bool ready = true;
#pragma unroll
  for (int x = 0; x < PT; ++x) {
    if (x >= (int)P) continue;
    const uint32_t c = P - 1 - x, bit = 1u << c;
    const uint32_t mask = (uint32_t)f[x] & ((1u << M) - 1), n = (uint32_t)(f[x] >> (M + pcb + 1));
    taken += n;
    uint64_t clk = (uint64_t)n * cfg.y;
    if ((f[x] >> (M + pcb)) & 1u) {
      const uint32_t full = (1u << (st[x].x & 0xFFFFu)) - 1u, lo = 32 - __clz(mask);
      const bool whole = mask == full, barrier = st[x].x & kBarrierBit;
      busy |= bit;
      clk = clk - cfg.y + st[x].y;
      if (mask || (st[x].x & kEnteredBit)) acted |= bit;
      ready = ready && whole && !barrier;
      if (whole && barrier) moves |= bit;          // passes its barrier
      marks |= ((full >> lo) << lo) << (c * M);    // PEs above the highest marked one
      if ((uint32_t)((f[x] >> M) & pc_mask) + 1 == S) leaving |= bit;
    }
    time = clk > time ? clk : time;
  }
  const uint32_t all = (1u << P) - 1u, left = cfg.x - taken;
  if ((cfg.z >> 31) && busy != all) {  // idle units that passed their last barrier at this time
#pragma unroll
    for (int x = 0; x < PT; ++x) {
      const uint32_t c = P - 1 - x, n = (uint32_t)(f[x] >> (M + pcb + 1));
      if (x < (int)P && !((busy >> c) & 1u) && n && (uint64_t)n * cfg.y == time) acted |= 1u << c;
    }
  }
  if (left) moves |= all & ~busy;  // dispatches
  const uint32_t h = acted ? 31 - __clz(acted) : 0u;  // the last unit that acted: earlier ones wait
  uint32_t slots = ((marks >> (h * M)) << (h * M)) | ((moves >> h) << (PM + h));
  if (busy && ready && !(left && busy != all) && !(prune && time + 1 > T)) slots |= 1u << (PM + P);
  // FIN (no work left, every unit idle) after the tick, or after the last
  // busy unit's barrier
  if (left == 0 && busy && (busy & ~leaving) == 0) {
    const bool tick = (slots >> (PM + P)) & 1u;
    const bool release = (busy & (busy - 1)) == 0 && ((slots >> PM) & busy);
    const uint64_t t = time + (tick ? 1 : 0);
    if ((tick || release) && t <= T) best = min(best, pack_tij(t, i, j));
  }
  return slots;
}

// The successor by `slot` of a state (its level field raised).
__device__ __forceinline__ u128 pe_succ(const PeParams& p, u128 key, uint32_t slot, uint32_t inv_M) {
  const uint32_t PM = p.P * p.M;
  u128 k = key + ((u128)1 << p.lvl_shift);
  if (slot < PM) {
    const uint32_t c = (slot * inv_M) >> 16;
    const uint32_t at = (p.P - 1 - c) * p.unit_bits + slot - c * p.M;
    return at < 64 ? k | (u128)(1ull << at) : k | ((u128)(1ull << (at - 64)) << 64);
  }
  // the tick moves every busy unit to its next step, a barrier its unit; a
  // dispatch takes a work-group
  const bool tick = slot == PM + p.P;
  const uint32_t i = (uint32_t)((uint64_t)(key >> p.wg_shift) & p.wg_mask) - 1;
  const uint32_t j = (uint32_t)((uint64_t)(key >> p.ts_shift) & p.ts_mask) - 1;
  const uint32_t S = __ldg(p.nsteps + i * p.b + j);
  for (uint32_t c = tick ? 0 : slot - PM; c < (tick ? p.P : slot - PM + 1); ++c) {
    const uint32_t shift = (p.P - 1 - c) * p.unit_bits;
    const Unit u = unpack(unit_field(key, p, c), p);
    if (u.busy) k ^= (u128)(pack(u, p) ^ pack(step_on(u, S), p)) << shift;
    else if (!tick) k += (u128)(3ull << (p.M + p.pc_bits)) << shift;  // n + 1, busy
  }
  return k;
}

// Position of set bit number k (from 0) of m; k < popc(m).
__device__ __forceinline__ uint32_t pe_nth_bit(uint32_t m, uint32_t k) {
  uint32_t pos = 0;
#pragma unroll
  for (uint32_t half = 16; half; half >>= 1) {
    const uint32_t c = __popc((m >> pos) & ((1u << half) - 1u));
    if (k >= c) {
      k -= c;
      pos += half;
    }
  }
  return pos;
}

// A warp's successors, dealt to its lanes: lane l writes numbers l, l + 32,
// ... of the `total` in the lanes' order; `upto` is the running count at each
// lane's end.
template <class Put>
__device__ __forceinline__ void pe_write(const PeParams& p, u128 key, uint32_t slots, uint32_t upto, uint32_t total,
                                         uint32_t lane, uint32_t inv_M, const Put& put) {
  for (uint32_t q0 = 0; q0 < total; q0 += 32) {
    const uint32_t q = q0 + lane;
    uint32_t o = 0;  // the lane whose state has successor q
#pragma unroll
    for (uint32_t step = 16; step; step >>= 1)
      if (__shfl_sync(0xffffffffu, upto, o + step - 1) <= q) o += step;
    o &= 31u;  // (beyond the total: any lane, nothing is written)
    const uint32_t his = __shfl_sync(0xffffffffu, slots, o);
    const uint32_t k = q - (__shfl_sync(0xffffffffu, upto, o) - __popc(his));
    const uint64_t lo = __shfl_sync(0xffffffffu, (unsigned long long)key, o);
    const uint64_t hi = __shfl_sync(0xffffffffu, (unsigned long long)(key >> 64), o);
    if (q < total) put(q, o, pe_succ(p, ((u128)hi << 64) | lo, pe_nth_bit(his, k), inv_M));
  }
}

// Running count over the warp's lanes (inclusive).
__device__ __forceinline__ uint32_t warp_upto(uint32_t v, uint32_t lane) {
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t w = __shfl_up_sync(0xffffffffu, v, o);
    if (lane >= (uint32_t)o) v += w;
  }
  return v;
}

template <int PT, bool SMALL>
__global__ void __launch_bounds__(kPeThreads, 2) pe_ordered_kernel(const __grid_constant__ PeArgs A) {
  extern __shared__ __align__(16) unsigned char pe_dyn[];
  PeSoloShared& solo = *reinterpret_cast<PeSoloShared*>(pe_dyn);
  const PeParams& p = A.p;
  Ctrl* ctrl = A.ctrl;
  const uint32_t tid = threadIdx.x, lane = tid & 31u, warp = tid >> 5, nw = blockDim.x >> 5;
  const uint64_t gtid = (uint64_t)blockIdx.x * blockDim.x + tid;
  const uint64_t nthreads = (uint64_t)gridDim.x * blockDim.x;
  __shared__ uint32_t s_cnt[kPeThreads / 32];
  __shared__ unsigned long long s_base, s_best, s_T;
  __shared__ uint32_t s_flags;
  uint32_t epoch = 0;
  const Barrier bar{A.bar, &A.ctrl->err, 0, A.timeout_ns};
  if (tid == 0) {
    s_T = A.T_src ? ld_relaxed_u64(A.T_src) + (uint64_t)A.T_delta : A.T;
    s_flags = 0;
    s_best = kNone;
  }
  __syncthreads();
  const uint64_t T = s_T;
  const bool prune = A.prune != 0;
  const uint64_t lpol = evict_first_policy();
  const uint32_t tb = A.tag_bits;
  const uint64_t tag = A.tag;

  // prologue: level arrays, levels 0..2 (the selects of Listing 3)
  for (uint64_t l = gtid; l < (uint64_t)p.max_level + 2; l += nthreads) {
    A.levels[2 * l] = l == 0 ? 1 : l == 1 ? p.a : l == 2 ? (uint64_t)p.a * p.b : 0;
    A.levels[2 * l + 1] = kNone;
    A.off[l] = l == 0 ? 0 : l == 1 ? 1 : l == 2 ? 1 + (uint64_t)p.a : 0;
  }
  {
    const uint64_t n_init = 1 + (uint64_t)p.a + (uint64_t)p.a * p.b;
    for (uint64_t x = gtid; x < n_init; x += nthreads) {
      u128 key = 0;
      uint32_t par = kNoParent;
      if (x >= 1 && x <= p.a) {
        key = ((u128)x << p.wg_shift) | ((u128)1 << p.lvl_shift);
        par = 0;
      } else if (x > p.a) {
        const uint64_t y = x - 1 - p.a;
        const uint32_t i = (uint32_t)(y / p.b), j = (uint32_t)(y % p.b);
        key = ((u128)(i + 1) << p.wg_shift) | ((u128)(j + 1) << p.ts_shift) | ((u128)2 << p.lvl_shift);
        par = i;
      }
      KeyOps<u128>::store(A.log_keys, x, LogTag<u128>::pack(key, tb, tag));
      A.log_par[x] = par;
    }
    if (gtid == 0) {
      ctrl->T = T;
      ctrl->best_pack = kNone;
      ctrl->wkey_lo = kNone;
      ctrl->wkey_hi = kNone;
      ctrl->widx = kNone;
    }
  }
  if (!grid_sync(bar, epoch)) return;

  // a log entry of this pass: tagged entries are loaded again until the tag
  // appears (bounded by the barrier timeout)
  auto entry = [&](uint64_t pos, u128 raw, u128& key) {
    key = raw;
    if (!tb || LogTag<u128>::unpack(key, tb, tag)) return true;
    const uint64_t t0 = globaltimer();
    for (;;) {
      __nanosleep(64);
      key = KeyOps<u128>::load(A.log_keys, pos);
      if (LogTag<u128>::unpack(key, tb, tag)) return true;
      if (globaltimer() - t0 > A.timeout_ns) {
        set_error(ctrl, MC_ERR_TIMEOUT);
        return false;
      }
    }
  };
  // places of a tile: every warp leaves its count in s_cnt, and after the
  // barrier sums the counts below its own, and all of them
  auto places = [&](uint32_t& total) {
    const uint32_t c = lane < nw ? s_cnt[lane] : 0u;
    total = __reduce_add_sync(0xffffffffu, c);
    return __reduce_add_sync(0xffffffffu, lane < warp ? c : 0u);
  };
  const uint32_t inv_M = 65536 / p.M + 1;  // slot / M by a multiplication (slots below 32)

  const uint32_t stop_mask = kPeFlagError | (A.early_exit ? kPeFlagViolation : 0u);
  uint32_t last = 2;
  uint64_t off_last = 1 + (uint64_t)p.a;
  uint64_t W = (uint64_t)p.a * p.b;
  uint64_t made = 0;  // successors of this block (thread 0)
  bool stop = false;
  for (; !stop;) {
    if (last >= p.max_level) break;
    if (W <= kPeSoloEnter) {
      // ---- block 0 alone, level after level in shared memory
      if (blockIdx.x == 0) {
        uint32_t L = last, cur = 0, n = (uint32_t)W, end = 0;
        uint64_t off = off_last;
        for (uint32_t x = tid; x < n; x += blockDim.x) {
          u128 key = 0;
          if (!entry(off + x, KeyOps<u128>::load(A.log_keys, off + x), key)) s_flags = kPeFlagError;
          solo.keys[0][x] = key;
        }
        __syncthreads();
        // an entry that never appeared is not a key: nothing decodes it, the
        // pass ends with the error that entry() set
        if (s_flags & kPeFlagError) end = 1;
        while (!end) {
          const uint64_t offN = off + n;
          uint64_t best = kNone;
          uint32_t done = 0;  // successors of the level so far
          for (uint32_t x0 = 0; x0 < n; x0 += blockDim.x) {
            const u128 key = x0 + tid < n ? solo.keys[cur][x0 + tid] : (u128)0;
            const uint32_t slots = x0 + tid < n ? pe_slots<PT, SMALL>(p, key, prune, T, best) : 0u;
            const uint32_t upto = warp_upto(__popc(slots), lane);
            const uint32_t wcnt = __shfl_sync(0xffffffffu, upto, 31);
            if (lane == 0) s_cnt[warp] = wcnt;
            if (best != kNone && x0 + blockDim.x >= n) atomicMin(&s_best, (unsigned long long)best);
            __syncthreads();
            uint32_t total;
            const uint32_t at = done + places(total);
            const uint32_t first = x0 + (tid & ~31u);
            pe_write(p, key, slots, upto, wcnt, lane, inv_M, [&](uint32_t q, uint32_t o, u128 succ) {
              const uint32_t to = at + q;
              if (to < kPeSoloCap) solo.keys[cur ^ 1][to] = succ;
              if (offN + to < A.log_cap) {
                LogIO<u128>::store(A.log_keys, offN + to, LogTag<u128>::pack(succ, tb, tag), lpol);
                st_u32_ef(A.log_par + offN + to, first + o, lpol);
              } else {
                s_flags = kPeFlagError;
              }
            });
            done += total;
            __syncthreads();  // the next tile rewrites the counts; the level's keys are complete
          }
          // (every thread sees the same totals and flags)
          const bool violated = s_best != kNone;
          if (tid == 0) {
            A.off[L + 1] = offN;
            A.levels[2 * (L + 1)] = done;
            if (violated) A.levels[2 * (L + 1) + 1] = s_best;
            made += done;
          }
          if (s_flags & kPeFlagError) {
            if (tid == 0) set_error(ctrl, MC_ERR_FRONTIER);
            end = 1;
          } else if (done == 0) {
            end = 1;
          } else {
            ++L;
            off = offN;
            n = done;
            cur ^= 1;
            if ((violated && A.early_exit) || L >= p.max_level) end = 1;
            else if (n > kPeSoloCap || (L & A.solo_mask) == 0) end = 2;  // back to every block
          }
          __syncthreads();
          if (tid == 0) s_best = kNone;
          __syncthreads();
        }
        if (tid == 0) {
          A.bar[kPeSoloLine * 32] = end;
          A.bar[kPeSoloLine * 32 + 1] = L;
        }
      }
      if (!grid_sync(bar, epoch)) return;
      const uint32_t end = ld_relaxed_u32(A.bar + kPeSoloLine * 32);
      last = ld_relaxed_u32(A.bar + kPeSoloLine * 32 + 1);
      off_last = ld_relaxed_u64(&A.off[last]);
      W = ld_relaxed_u64(A.levels + 2 * last) & kLevelWidthMask;
      stop = end == 1;
      continue;
    }
    // ---- every block
    const uint32_t L = last;
    const uint64_t offN = off_last + W;
    if (gtid == 0) A.off[L + 1] = offN;
    uint64_t* lvl_next = A.levels + 2 * (L + 1);
    const uint32_t Wl = (uint32_t)W, threads = (uint32_t)nthreads;
    const uint32_t R = Wl > threads ? kPeKeys : 1;
    const uint32_t stride = threads * R;
    uint32_t base = blockIdx.x * blockDim.x * R + tid;
    uint64_t best = kNone;
    // (a block without a state of the level only arrives)
    bool more = base - tid < Wl;
    if (!more && tb && tid == 0) (void)level_arrive_reserve(lvl_next, &s_flags, stop_mask, 0);
    while (more) {
      more = base - tid + stride < Wl;  // (uniform: the block's tiles end together)
      PeOwn own[kPeKeys];
      u128 raw[kPeKeys];
#pragma unroll
      for (int r = 0; r < kPeKeys; ++r)
        if (r < (int)R && base + r * blockDim.x < Wl)
          raw[r] = LogIO<u128>::load(A.log_keys, off_last + base + r * blockDim.x, lpol);
      uint32_t upto[kPeKeys], row[kPeKeys], wcnt = 0;  // running counts and totals of the warp's rows
#pragma unroll
      for (int r = 0; r < kPeKeys; ++r) {
        const uint32_t s = base + r * blockDim.x;
        own[r].slots = 0;
        own[r].key = 0;
        upto[r] = row[r] = 0;
        if (r >= (int)R) continue;
        if (s < Wl) {
          if (entry(off_last + s, raw[r], own[r].key)) own[r].slots = pe_slots<PT, SMALL>(p, own[r].key, prune, T, best);
          else atomicOr(&s_flags, kPeFlagError);
        }
        upto[r] = warp_upto(__popc(own[r].slots), lane);
        row[r] = __shfl_sync(0xffffffffu, upto[r], 31);
        wcnt += row[r];
      }
      if (lane == 0) s_cnt[warp] = wcnt;
      if (!more && best != kNone) atomicMin(&s_best, (unsigned long long)best);
      __syncthreads();
      uint32_t total;
      const uint32_t before = places(total);
      if (tid == 0) {
        if (!more && s_best != kNone) {
          atomicMin(reinterpret_cast<unsigned long long*>(lvl_next + 1), s_best);
          s_best = kNone;
          atomicOr(&s_flags, kPeFlagViolation);
        }
        if (!more && tb) s_base = level_arrive_reserve(lvl_next, &s_flags, stop_mask, total);
        else s_base = total ? level_reserve(lvl_next, total) : 0ull;
        made += total;
        // a level's width is counted in 32 bits: a level of 2^31 states ends
        // the query (each block is at most one tile beyond)
        if (s_base >= (1ull << 31)) set_error(ctrl, MC_ERR_FRONTIER);
      }
      __syncthreads();
      if (s_base >= (1ull << 31)) {
        atomicOr(&s_flags, kPeFlagError);
        if (more && tb && tid == 0)  // arrive without the tiles that are left
          (void)level_arrive_reserve(lvl_next, &s_flags, stop_mask, 0);
        more = false;
      } else if (wcnt) {
        uint64_t at0 = offN + s_base + before;
        if (at0 + wcnt <= A.log_cap) {
#pragma unroll
          for (int r = 0; r < kPeKeys; ++r) {
            if (r >= (int)R) continue;
            const uint32_t first = base - lane + r * blockDim.x;
            pe_write(p, own[r].key, own[r].slots, upto[r], row[r], lane, inv_M, [&](uint32_t q, uint32_t o, u128 succ) {
              LogIO<u128>::store(A.log_keys, at0 + q, LogTag<u128>::pack(succ, tb, tag), lpol);
              st_u32_ef(A.log_par + at0 + q, first + o, lpol);
            });
            at0 += row[r];
          }
        } else if (lane == 0) {  // beyond the log's capacity: nothing is written, the pass fails
          set_error(ctrl, MC_ERR_FRONTIER);
          atomicOr(&s_flags, kPeFlagError);
        }
      }
      base += stride;
    }
    uint64_t word = 0;
    if (!(tb ? level_wait(bar, lvl_next, &word) : level_sync(bar, lvl_next, &s_flags, stop_mask, &word))) return;
    const uint64_t Wn = word & kLevelWidthMask;
    if (offN + Wn > A.log_cap) {  // the same decision in every block (one final word)
      set_error(ctrl, MC_ERR_FRONTIER);
      break;
    }
    if ((word >> kLevelStopShift) & 0xFFFFu) {
      if (ld_relaxed_u32(&ctrl->err)) break;
      last = L + 1;
      off_last = offN;
      W = Wn;
      break;
    }
    if (Wn == 0) break;
    last = L + 1;
    off_last = offN;
    W = Wn;
  }
  if (tid == 0 && made)
    atomicAdd(reinterpret_cast<unsigned long long*>(&ctrl->probes), (unsigned long long)made);
  if (ld_relaxed_u32(&ctrl->err)) return;

  // first level holding a violating FIN state, and the minimum over all levels
  uint32_t wl = 0;
  uint64_t best_all = kNone;
  if (A.early_exit) {
    best_all = ld_relaxed_u64(A.levels + 2 * last + 1);
    wl = best_all != kNone ? last : 0;
  } else {
    __shared__ unsigned int s_wl;
    if (tid == 0) {
      s_best = kNone;
      s_wl = 0xFFFFFFFFu;
    }
    __syncthreads();
    for (uint32_t l = 3 + tid; l <= last; l += blockDim.x) {
      const uint64_t b = ld_relaxed_u64(A.levels + 2 * l + 1);
      if (b != kNone) {
        atomicMin(&s_best, (unsigned long long)b);
        atomicMin(&s_wl, l);
      }
    }
    __syncthreads();
    best_all = s_best;
    wl = s_wl == 0xFFFFFFFFu ? 0 : s_wl;
  }
  if (gtid == 0) {
    ctrl->levels = last + 1;
    ctrl->states = off_last + W;
    ctrl->stop_level = wl;
    ctrl->best_pack = best_all;
    ctrl->wpack = wl ? ld_relaxed_u64(A.levels + 2 * wl + 1) : kNone;
    if (A.tmin_out && best_all != kNone) *A.tmin_out = pack_time(best_all);
  }
  if (!A.want_witness || wl == 0) return;

  // witness: among the FIN states of level wl with the level's minimum
  // (time, i, j), the smallest key (high word first, then low word)
  const uint64_t target = ld_relaxed_u64(A.levels + 2 * wl + 1);
  const uint64_t offW = ld_relaxed_u64(&A.off[wl]);
  const uint64_t Ww = ld_relaxed_u64(A.levels + 2 * wl) & kLevelWidthMask;
  auto matches = [&](u128 key) {
    Decoded d;
    decode(key, p, d);
    return is_fin(d) && pack_tij(d.time, d.i, d.j) == target;
  };
  for (uint64_t x = gtid; x < Ww; x += nthreads) {
    u128 key;
    if (!entry(offW + x, KeyOps<u128>::load(A.log_keys, offW + x), key)) break;
    if (matches(key))
      atomicMin(reinterpret_cast<unsigned long long*>(&ctrl->wkey_hi), (unsigned long long)(key >> 64));
  }
  if (!grid_sync(bar, epoch)) return;
  const uint64_t whi = ld_relaxed_u64(&ctrl->wkey_hi);
  for (uint64_t x = gtid; x < Ww; x += nthreads) {
    u128 key;
    if (!entry(offW + x, KeyOps<u128>::load(A.log_keys, offW + x), key)) break;
    if ((uint64_t)(key >> 64) == whi && matches(key))
      atomicMin(reinterpret_cast<unsigned long long*>(&ctrl->wkey_lo), (unsigned long long)key);
  }
  if (!grid_sync(bar, epoch)) return;
  {
    const uint64_t wlo = ld_relaxed_u64(&ctrl->wkey_lo);
    for (uint64_t x = gtid; x < Ww; x += nthreads) {
      u128 key;
      if (!entry(offW + x, KeyOps<u128>::load(A.log_keys, offW + x), key)) break;
      if ((uint64_t)key == wlo && (uint64_t)(key >> 64) == whi) ctrl->widx = x;
    }
  }
  if (!grid_sync(bar, epoch)) return;
  if (gtid == 0) {
    uint64_t idx = ld_relaxed_u64(&ctrl->widx);
    if (idx >= Ww) {
      set_error(ctrl, MC_ERR_FRONTIER);
      return;
    }
    uint64_t off = offW;
    for (uint32_t l = wl;; --l) {
      const uint64_t at = off + idx;
      const u128 raw = KeyOps<u128>::load(A.log_keys, at);
      const uint32_t par = __ldcg(A.log_par + at);
      if (l) off = ld_relaxed_u64(&A.off[l - 1]);  // in flight together
      u128 key;
      if (!entry(at, raw, key)) return;
      A.trace[2 * l] = (uint64_t)key;
      A.trace[2 * l + 1] = (uint64_t)(key >> 64);
      if (l == 0) break;
      idx = par;
    }
    ctrl->witness_level = wl;
    ctrl->trace_len = wl + 1;
  }
}

const void* pe_ordered_pick(const PeParams& p) {
  if (p.unit_bits > 32)
    return p.P <= 4 ? (const void*)pe_ordered_kernel<4, false> : (const void*)pe_ordered_kernel<8, false>;
  return p.P <= 4 ? (const void*)pe_ordered_kernel<4, true> : (const void*)pe_ordered_kernel<8, true>;
}

}  // namespace
}  // namespace mc
