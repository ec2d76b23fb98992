// Ordered expansion: the level engine's pass for FREE models whose insert is
// left to the library (mc_options.probe_scheme AUTO).
//
// Under FREE any unit may take the next work-group, so a state is reached
// from as many predecessors as units have started, and the general pass
// (mc_explore.cuh) proposes it that many times to the visited set.  Here a
// state proposes unit c only when no unit above c has started yet.  Every
// state is still generated, at its level, and exactly once: its last unit
// with a work-group, c, names the one state that proposes it, the state
// without one work-group of c.  That state was kept, because clocks only grow
// (what pruning keeps is closed under taking a work-group back), so by
// induction the kept states of every level are those of the general pass.
// A state that is generated once needs no visited set: no table is
// allocated, cleared or probed.
//
// The frontier log, the level records, the level barrier fused with the width
// counter and the tagged log entries are those of the general pass.  The log's
// parent indices are neither written nor read: a state's counts name its path
// (all work-groups of unit 0, then unit 1's, ...), so the trace is built from
// the witness, a level per thread, and the witness's place is not looked up.
//
// What bounds it: on wide levels the log, each key written once and read once
// by the next level (32 bytes a state with 128-bit keys: C3 at G=36 moves 5.1
// of the 6.8 TB/s a copy reaches, the rest waits at the tiles' barriers; a
// query takes 6.85 ms, and took 7.14 with parent indices written, 36 bytes);
// on narrow ones the chain of a level (key load, reservation fused with the
// arrival, poll; 3.4 us a level on C2 at G=80).  A tile is blockDim x R keys,
// R up to kTreeKeys, so that one reservation (an atomic on the level's one
// word) covers a thousand states; the next tile's keys are loaded before the
// reservation is waited for.  In a level with fewer states than threads a
// tile is one key per thread.  Measured on C3 at G=28 (with parent indices):
// 4 keys per thread and 4 blocks of 256 per SM 1.37 ms, 2 blocks of 512 1.39,
// 8 of 128 1.40; 6 keys spill, 6 blocks (40 registers) 1.87.
#include "mc_explore.cuh"
#include "mc_tree.h"

namespace mc {
namespace {

using namespace mc::dev;

constexpr int kTreeKeys = 4;
constexpr uint32_t kTreeTable = 1024;  // work-group counts by (i, j) field kept in shared memory

template <class A>
__device__ __forceinline__ uint32_t lowest_bit(A x);
template <>
__device__ __forceinline__ uint32_t lowest_bit<uint64_t>(uint64_t x) { return (uint32_t)__ffsll((long long)x) - 1; }
template <>
__device__ __forceinline__ uint32_t lowest_bit<u128>(u128 x) {
  return (uint64_t)x ? lowest_bit((uint64_t)x) : 64 + lowest_bit((uint64_t)(x >> 64));
}

// How a key is stored in the log: tagged with the pass in the top `tag_bits`
// of its words (8 to 16; see the general pass), or as it is.
//   64-bit words       the tag above the key;
//   128-bit words with keys computed in 64 bits (at most 56 used): the low
//                      word the same, the high word all tag;
//   128-bit keys       as the general pass stores them.
// The tag of a 64-bit word is compared and taken off by one exclusive or of
// its upper half.
template <class K, class A>
struct TreeLog;

__device__ __forceinline__ bool strip_tag(uint64_t w, uint32_t tag_hi, uint32_t most, uint64_t& key) {
  const uint32_t hi = (uint32_t)(w >> 32) ^ tag_hi;
  key = ((uint64_t)hi << 32) | (uint32_t)w;
  return hi <= most;
}

template <>
struct TreeLog<uint64_t, uint64_t> {
  // the tag in a word's upper half; the most that half of a key can be (all
  // ones without a tag: a key of 64 used bits may have them all set)
  uint32_t tag_hi, most;
  __device__ TreeLog(uint32_t tb, uint64_t tag) : tag_hi(tb ? (uint32_t)tag << (32 - tb) : 0u),
                                                  most(0xFFFFFFFFu >> tb) {}
  __device__ uint64_t pack(uint64_t k) const { return k | ((uint64_t)tag_hi << 32); }
  __device__ bool unpack(uint64_t w, uint64_t& key) const { return strip_tag(w, tag_hi, most, key); }
};

template <>
struct TreeLog<u128, uint64_t> {
  uint32_t tag_hi, most;
  uint64_t high;
  __device__ TreeLog(uint32_t tb, uint64_t tag) : tag_hi(tb ? (uint32_t)tag << (32 - tb) : 0u),
                                                  most(0xFFFFFFFFu >> tb), high(tb ? tag : 0) {}
  __device__ u128 pack(uint64_t k) const { return ((u128)high << 64) | k | ((uint64_t)tag_hi << 32); }
  __device__ bool unpack(u128 w, uint64_t& key) const {
    return strip_tag((uint64_t)w, tag_hi, most, key) && (uint64_t)(w >> 64) == high;
  }
};

template <>
struct TreeLog<u128, u128> {
  uint32_t tb;
  uint64_t tag;
  __device__ TreeLog(uint32_t b, uint64_t t) : tb(b), tag(t) {}
  __device__ u128 pack(u128 k) const { return LogTag<u128>::pack(k, tb, tag); }
  __device__ bool unpack(u128 w, u128& key) const {
    key = w;
    return tb == 0 || LogTag<u128>::unpack(key, tb, tag);
  }
};

// The key of log entry `pos` from a first load: in a tagged log, loaded again
// until it carries this pass's tag.  False (and MC_ERR_TIMEOUT) when it does
// not appear within the barrier timeout.
template <class K, class A>
__device__ __forceinline__ bool tree_entry(const ExploreArgs& G, const TreeLog<K, A>& log, uint64_t pos, K raw, A& key) {
  if (log.unpack(raw, key)) return true;
  const uint64_t t0 = globaltimer();
  for (;;) {
    __nanosleep(64);
    if (log.unpack(KeyOps<K>::load(G.log_keys, pos), key)) return true;
    if (globaltimer() - t0 > G.timeout_ns) {
      set_error(G.ctrl, MC_ERR_TIMEOUT);
      key = 0;
      return false;
    }
  }
}

// The successors' times of a state whose lowest nonzero count field is f0:
// max(the state's time, the starting unit's next clock).  PRUNE: takes the
// units whose successor passes T out of `starts`.  When the successors are
// terminal (FIN, Listing 4), those within T violate G(FIN -> time > T) (Step
// 2), and the least of them lowers `best`.  The units of the fields below f0
// have not started, so their next clocks are one work-group each; `least[f]`
// is the least speed of the fields below f (2^32 - 1 for f = 0).  Clocks in C:
// 32 bits when every clock of the model fits.  (One state in five has terminal
// successors on C3 at G=36: with a loop per field and per successor in 64 bits
// this was 40% of the pass.)
template <bool PRUNE, class C, class A>
__device__ __forceinline__ void tree_times(const Params& p, A key, uint32_t f0, uint64_t cost, bool terminal,
                                           uint64_t T, uint32_t i, uint32_t j, const uint32_t* speed,
                                           const uint32_t* least, uint32_t& starts, uint64_t& best) {
  const uint32_t mask = (uint32_t)p.n_mask;
  C mx = 0;
  A x = key;
  for (uint32_t f = 0; f < p.P; f += 4) {  // (speeds beyond P are 0)
    const uint4 s = *reinterpret_cast<const uint4*>(speed + f);
    const C c0 = (C)((uint32_t)x & mask) * s.x;
    x >>= p.n_bits;
    const C c1 = (C)((uint32_t)x & mask) * s.y;
    x >>= p.n_bits;
    const C c2 = (C)((uint32_t)x & mask) * s.z;
    x >>= p.n_bits;
    const C c3 = (C)((uint32_t)x & mask) * s.w;
    x >>= p.n_bits;
    mx = max(max(mx, max(c0, c1)), max(c2, c3));
  }
  const C own = (C)(((uint32_t)(key >> (f0 * p.n_bits)) & mask) + 1) * speed[f0];
  if (PRUNE) {
    if ((uint64_t)max(mx, own) * cost > T) starts &= ~(1u << f0);
    for (uint32_t f = 0; f < f0; ++f)
      if ((uint64_t)max(mx, (C)speed[f]) * cost > T) starts &= ~(1u << f);
  }
  if (terminal) {
    // (no field below the lowest: least[0] is beyond every clock of 32 bits,
    // but not of 64)
    const C other = sizeof(C) == 8 && f0 == 0 ? (C)~(C)0 : (C)least[f0];
    const uint64_t t = (uint64_t)max(mx, min(own, other)) * cost;
    if (t <= T && t <= pack_time(best)) best = min(best, pack_tij(t, i, j));
  }
}

template <class K, class A, bool PRUNE>
__global__ void __launch_bounds__(kTreeThreads, 4) tree_kernel(const __grid_constant__ ExploreArgs G) {
  const Params& p = G.p;
  Ctrl* ctrl = G.ctrl;
  const uint32_t tid = threadIdx.x, lane = tid & 31u, warp = tid >> 5, nw = blockDim.x >> 5;
  const uint64_t gtid = (uint64_t)blockIdx.x * blockDim.x + tid;
  const uint64_t nthreads = (uint64_t)gridDim.x * blockDim.x;
  __shared__ uint32_t s_cnt[kTreeThreads / 32];
  __shared__ unsigned long long s_base, s_best, s_T;
  __shared__ uint32_t s_flags, s_skip;
  __shared__ __align__(16) uint32_t s_speed[kMaxP];  // by field: unit P-1-f
  __shared__ uint32_t s_least[kMaxP];                // the least speed of the fields below
  __shared__ uint32_t s_N[kTreeTable];
  uint32_t epoch = 0;  // device-wide barriers passed in this pass
  const Barrier bar{G.bar_lines, &G.ctrl->err, G.barrier_extra, G.timeout_ns};

  // the threshold, as in the general pass: given, read from the device, or
  // one below the chained predecessor's counterexample time
  if (tid == 0) {
    uint64_t t = G.T;
    uint32_t skip = 0;
    if (G.T_src) t = ld_relaxed_u64(G.T_src) + (uint64_t)G.T_delta;
    if (G.prev) {
      const Ctrl* q = G.prev;
      if (ld_relaxed_u32(&q->err) || ld_relaxed_u32(&q->skipped) || ld_relaxed_u32(&q->stop_level) == 0) skip = 1;
      else t = pack_time(ld_relaxed_u64(&q->wpack)) - 1;
    }
    s_T = t;
    s_skip = skip;
    s_flags = 0;
    s_best = kNone;
  }
  if (warp == 0) {
    const uint32_t own = lane < p.P ? __ldg(p.speed + p.P - 1 - lane) : 0u;
    uint32_t least = __shfl_up_sync(0xffffffffu, own, 1);
#pragma unroll
    for (uint32_t o = 1; o < kMaxP; o <<= 1) {
      const uint32_t v = __shfl_up_sync(0xffffffffu, least, o);
      if (lane > o) least = min(least, v);
    }
    if (lane < kMaxP) {
      s_speed[lane] = own;
      s_least[lane] = lane ? least : 0xFFFFFFFFu;
    }
  }
  // N_ij by the key's (i, j) bits, one lookup per state instead of two fields
  // and a gather; larger domains read the table in global memory
  const uint32_t ts_bits = p.wg_shift - p.ts_shift;
  const bool small = ((uint64_t)(p.a + 1) << ts_bits) <= kTreeTable;
  if (small)
    for (uint32_t x = tid; x < p.a * p.b; x += blockDim.x)
      s_N[((x / p.b + 1) << ts_bits) | (x % p.b + 1)] = __ldg(p.N + x);
  // lowest nonzero count field = lowest set bit / n_bits, by a multiplication
  // (exact for bits below 128 and fields of at most 32 bits)
  const uint32_t inv_bits = 65536 / p.n_bits + 1;
  const A counts = ((A)1 << (p.P * p.n_bits)) - 1;
  const uint32_t mask0 = (uint32_t)p.n_mask;
  __syncthreads();
  if (s_skip) {
    if (gtid == 0) ctrl->skipped = 1;
    return;
  }
  const uint64_t T = s_T;
  const TreeLog<K, A> log(G.tag_bits, G.tag);
  const uint64_t lpol = evict_first_policy();

  // prologue: level arrays, levels 0..2 (the selects, Listing 3)
  for (uint64_t l = gtid; l < (uint64_t)p.max_level + 2; l += nthreads) {
    G.levels[2 * l] = l == 0 ? 1 : l == 1 ? p.a : l == 2 ? (uint64_t)p.a * p.b : 0;
    G.levels[2 * l + 1] = kNone;
    G.off[l] = l == 0 ? 0 : l == 1 ? 1 : l == 2 ? 1 + (uint64_t)p.a : 0;
  }
  {
    const uint64_t n_init = 1 + (uint64_t)p.a + (uint64_t)p.a * p.b;
    for (uint64_t x = gtid; x < n_init; x += nthreads) {
      A key = 0;
      if (x >= 1 && x <= p.a) {
        key = (A)x << p.wg_shift;
      } else if (x > p.a) {
        const uint64_t y = x - 1 - p.a;
        key = ((A)(y / p.b + 1) << p.wg_shift) | ((A)(y % p.b + 1) << p.ts_shift);
      }
      KeyOps<K>::store(G.log_keys, x, log.pack(key));
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

  // level loop (one device-wide barrier per level)
  const uint32_t stop_mask = kFlagError | (G.early_exit ? kFlagViolation : 0u);
  uint32_t last = 2;
  uint64_t off_last = 1 + (uint64_t)p.a;
  uint64_t W = (uint64_t)p.a * p.b;
  for (;;) {
    const uint32_t L = last;
    if (L >= p.max_level) break;  // the deepest level holds only terminals
    const uint64_t offN = off_last + W;
    if (gtid == 0) G.off[L + 1] = offN;
    uint64_t* lvl_next = G.levels + 2 * (L + 1);
    const uint32_t k_cur = L - 2;  // work-groups taken at level L
    // (a level is narrower than 2^31 states: 32-bit indexes inside it)
    const uint32_t Wl = (uint32_t)W, threads = (uint32_t)nthreads;
    const uint32_t per = (Wl + threads - 1) / threads;
    const uint32_t R = per < kTreeKeys ? per : (uint32_t)kTreeKeys;
    const uint32_t stride = threads * R;
    uint32_t base = blockIdx.x * blockDim.x * R + tid;  // this thread's first state of the tile
    uint64_t best = kNone;
    const K* const src = reinterpret_cast<const K*>(G.log_keys) + off_last;
    K raw[kTreeKeys];
#pragma unroll
    for (int r = 0; r < kTreeKeys; ++r)
      if (r < (int)R && base + r * blockDim.x < Wl) raw[r] = LogIO<K>::load(src, base + r * blockDim.x, lpol);
    // (a block without a state of the level only arrives)
    bool more = base - tid < Wl;
    if (!more && G.tag_bits && tid == 0) (void)level_arrive_reserve(lvl_next, &s_flags, stop_mask, 0);
    while (more) {
      more = base - tid + stride < Wl;  // (uniform: the block's tiles end together)
      A key[kTreeKeys];
      // which units start: field f of the key (at f * n_bits) is unit P-1-f.
      // PRUNE: bit f; else the number of them, a run of fields from 0
      uint32_t starts[kTreeKeys];
      uint32_t cnt = 0;       // this lane's successors (not PRUNE: by other units than the last)
      uint32_t by_last = 0;   // not PRUNE: the warp's successors by the last unit
#pragma unroll
      for (int r = 0; r < kTreeKeys; ++r) {
        const uint32_t s = base + r * blockDim.x;
        starts[r] = 0;
        key[r] = 0;
        if (r >= (int)R) continue;
        uint32_t ij = 0, left = 0;
        if (s < Wl) {
          if (tree_entry(G, log, off_last + s, raw[r], key[r])) {
            ij = (uint32_t)(key[r] >> p.ts_shift);
            left = (small ? s_N[ij] : __ldg(p.N + ((ij >> ts_bits) - 1) * p.b + (ij & p.ts_mask) - 1)) - k_cur;
          } else {
            atomicOr(&s_flags, kFlagError);
          }
        }
        // every unit from the last started one on (all of them from a
        // select); most states have started the last unit, most rows of 32
        // have only such
        const bool alive = left != 0;
        const uint32_t m = __ballot_sync(0xffffffffu, alive);
        if (!m) continue;  // 32 terminal states, or none
        uint32_t f0 = 0;
        if (__any_sync(0xffffffffu, alive && ((uint32_t)key[r] & mask0) == 0)) {
          const A x = key[r] & counts;
          f0 = !alive ? 0u : x ? (lowest_bit<A>(x) * inv_bits) >> 16 : p.P - 1;
        }
        starts[r] = !alive ? 0u : PRUNE ? (2u << f0) - 1u : f0 + 1;
        if (alive && (PRUNE || left == 1)) {
          const uint32_t i = (ij >> ts_bits) - 1, j = (ij & p.ts_mask) - 1;
          const uint64_t cost = __ldg(p.cost + i * p.b + j);
          if (p.clk32) tree_times<PRUNE, uint32_t>(p, key[r], f0, cost, left == 1, T, i, j, s_speed, s_least, starts[r], best);
          else tree_times<PRUNE, uint64_t>(p, key[r], f0, cost, left == 1, T, i, j, s_speed, s_least, starts[r], best);
        }
        if (PRUNE) {
          cnt += __popc(starts[r]);
        } else {
          cnt += f0;
          by_last += __popc(m);
        }
      }
      // the next tile's keys are on their way while this tile's places are
      // reserved and its successors written
      base += stride;
      if (more) {
#pragma unroll
        for (int r = 0; r < kTreeKeys; ++r)
          if (r < (int)R && base + r * blockDim.x < Wl) raw[r] = LogIO<K>::load(src, base + r * blockDim.x, lpol);
      }
      const uint32_t wcnt = by_last + (__any_sync(0xffffffffu, cnt) ? __reduce_add_sync(0xffffffffu, cnt) : 0u);
      if (lane == 0) s_cnt[warp] = wcnt;
      if (!more && best != kNone) atomicMin(&s_best, (unsigned long long)best);
      __syncthreads();
      // every warp sums the counts below its own, and all of them
      const uint32_t wc = lane < nw ? s_cnt[lane] : 0u;
      const uint32_t total = __reduce_add_sync(0xffffffffu, wc);
      const uint32_t before = __reduce_add_sync(0xffffffffu, lane < warp ? wc : 0u);
      if (tid == 0) {
        if (!more && s_best != kNone) {
          atomicMin(reinterpret_cast<unsigned long long*>(lvl_next + 1), s_best);
          s_best = kNone;
          atomicOr(&s_flags, kFlagViolation);
        }
        // the block's last tile of a tagged log: the reservation is the
        // block's arrival at the level barrier
        if (!more && G.tag_bits) s_base = level_arrive_reserve(lvl_next, &s_flags, stop_mask, total);
        else s_base = total ? level_reserve(lvl_next, total) : 0ull;
      }
      __syncthreads();
      if (wcnt) {
        const uint64_t at0 = offN + s_base + before;
        if (at0 + wcnt <= G.log_cap) {
          K* const dst = reinterpret_cast<K*>(G.log_keys) + at0;
          const uint32_t below = (1u << lane) - 1u;
          auto put = [&](uint32_t& at, bool mine, A succ) {  // a warp's stores are consecutive
            const uint32_t m = __ballot_sync(0xffffffffu, mine);
            if (mine) LogIO<K>::store(dst, at + __popc(m & below), log.pack(succ), lpol);
            at += __popc(m);
          };
          // the last unit's successors first, the others behind them: rows
          // of the next level then rarely hold both kinds
          uint32_t at = 0, other = by_last;
#pragma unroll
          for (int r = 0; r < kTreeKeys; ++r) {
            if (r >= (int)R) continue;
            if (PRUNE) {
              for (uint32_t any = __reduce_or_sync(0xffffffffu, starts[r]); any; any &= any - 1) {
                const uint32_t f = __ffs(any) - 1;
                put(at, (starts[r] >> f) & 1u, key[r] + ((A)1 << (f * p.n_bits)));
              }
            } else {
              put(at, starts[r] != 0, key[r] + 1);
              A one = (A)1 << p.n_bits;
              for (uint32_t f = 1; __any_sync(0xffffffffu, f < starts[r]); ++f, one <<= p.n_bits)
                put(other, f < starts[r], key[r] + one);
            }
          }
        } else if (lane == 0) {  // beyond the log's capacity: nothing is written, the query fails
          set_error(ctrl, MC_ERR_FRONTIER);
          atomicOr(&s_flags, kFlagError);
        }
      }
    }
    // level L+1's width word doubles as the barrier (see the general pass)
    uint64_t word = 0;
    if (!(G.tag_bits ? level_wait(bar, lvl_next, &word) : level_sync(bar, lvl_next, &s_flags, stop_mask, &word)))
      return;
    const uint64_t Wn = word & kLevelWidthMask;
    if (offN + Wn > G.log_cap) {  // the same decision in every block (one final word)
      set_error(ctrl, MC_ERR_FRONTIER);
      break;
    }
    if ((word >> kLevelStopShift) & 0xFFFFu) {  // an error, or level L+1 holds a violating terminal
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
  if (ld_relaxed_u32(&ctrl->err)) return;

  // first level holding a violating terminal, and the minimum over all levels
  uint32_t wl = 0;
  uint64_t best_all = kNone;
  if (G.early_exit) {
    best_all = ld_relaxed_u64(G.levels + 2 * last + 1);
    wl = best_all != kNone ? last : 0;
  } else {
    __shared__ unsigned int s_wl;
    if (tid == 0) {
      s_best = kNone;
      s_wl = 0xFFFFFFFFu;
    }
    __syncthreads();
    for (uint32_t l = 3 + tid; l <= last; l += blockDim.x) {
      const uint64_t b = ld_relaxed_u64(G.levels + 2 * l + 1);
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
    ctrl->wpack = wl ? ld_relaxed_u64(G.levels + 2 * wl + 1) : kNone;
    if (G.tmin_out && best_all != kNone) *G.tmin_out = pack_time(best_all);
  }
  if (!G.want_witness || wl == 0) return;

  // witness: the violating terminal of level wl with the smallest key among
  // those with the level's minimum (time, i, j)
  const uint64_t target = ld_relaxed_u64(G.levels + 2 * wl + 1);
  const uint64_t offW = ld_relaxed_u64(&G.off[wl]);
  const uint64_t Ww = ld_relaxed_u64(G.levels + 2 * wl) & kLevelWidthMask;
  const uint32_t ti = pack_i(target), tj = pack_j(target);
  const uint64_t tt = pack_time(target);
  const uint32_t cfg_t = ti * p.b + tj;
  const uint32_t n_t = __ldg(p.N + cfg_t);
  auto matches = [&](A key) {
    return field(key, p.wg_shift, p.wg_mask) - 1 == ti && field(key, p.ts_shift, p.ts_mask) - 1 == tj &&
           sum_n(key, p) == n_t && key_time(key, p, cfg_t) == tt;
  };
  unsigned long long* const wlo = reinterpret_cast<unsigned long long*>(&ctrl->wkey_lo);
  unsigned long long* const whi = reinterpret_cast<unsigned long long*>(&ctrl->wkey_hi);
  for (uint64_t x = gtid; x < Ww; x += nthreads) {
    A key;
    if (!tree_entry(G, log, offW + x, KeyOps<K>::load(G.log_keys, offW + x), key)) break;
    if (!matches(key)) continue;
    if (sizeof(A) == 8) atomicMin(wlo, (unsigned long long)key);
    else atomicMin(whi, (unsigned long long)KeyOps<A>::hi(key));
  }
  if (!grid_sync(bar, epoch)) return;
  if (sizeof(A) == 16) {
    const uint64_t hi = ld_relaxed_u64(&ctrl->wkey_hi);
    for (uint64_t x = gtid; x < Ww; x += nthreads) {
      A key;
      if (!tree_entry(G, log, offW + x, KeyOps<K>::load(G.log_keys, offW + x), key)) break;
      if (KeyOps<A>::hi(key) == hi && matches(key)) atomicMin(wlo, (unsigned long long)KeyOps<A>::lo(key));
    }
    if (!grid_sync(bar, epoch)) return;
  }
  // the trace s0 -> the witness, in the order in which states are generated
  if (blockIdx.x) return;
  const uint64_t lo = ld_relaxed_u64(&ctrl->wkey_lo), hi = sizeof(A) == 16 ? ld_relaxed_u64(&ctrl->wkey_hi) : 0;
  if (lo == kNone || (sizeof(A) == 16 && hi == kNone)) {  // cannot happen when the level is intact
    if (tid == 0) set_error(ctrl, MC_ERR_FRONTIER);
    return;
  }
  const A witness = sizeof(A) == 16 ? (A)(((u128)hi << 64) | lo) : (A)lo;
  for (uint32_t l = tid; l <= wl; l += blockDim.x) {
    A key = l >= 1 ? (A)(ti + 1) << p.wg_shift : (A)0;
    if (l >= 2) {
      key |= (A)(tj + 1) << p.ts_shift;
      uint32_t rest = l - 2;
      for (uint32_t u = 0; u < p.P; ++u) {
        const uint32_t shift = (p.P - 1 - u) * p.n_bits, n = min(rest, (uint32_t)field(witness, shift, p.n_mask));
        key |= (A)n << shift;
        rest -= n;
      }
    }
    G.trace[2 * l] = KeyOps<A>::lo(key);
    G.trace[2 * l + 1] = KeyOps<A>::hi(key);
  }
  if (tid == 0) {
    if (sizeof(A) == 8) ctrl->wkey_hi = 0;
    ctrl->witness_level = wl;
    ctrl->trace_len = wl + 1;
  }
}

template <class K, class A>
const void* pick_prune(bool prune) {
  return prune ? (const void*)tree_kernel<K, A, true> : (const void*)tree_kernel<K, A, false>;
}

const void* pick_tree(int key_words, uint32_t used_bits, bool prune) {
  if (key_words == 1) return pick_prune<uint64_t, uint64_t>(prune);
  return used_bits <= kTreeNarrow ? pick_prune<u128, uint64_t>(prune) : pick_prune<u128, u128>(prune);
}

}  // namespace

// (of the two kernels of a model, with and without pruning, the smaller)
int tree_occupancy(int key_words, uint32_t used_bits, int threads, int* blocks_per_sm) {
  *blocks_per_sm = 1 << 20;
  for (int prune = 0; prune < 2; ++prune) {
    int n = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, pick_tree(key_words, used_bits, prune), threads, 0) !=
        cudaSuccess)
      return -1;
    *blocks_per_sm = n < *blocks_per_sm ? n : *blocks_per_sm;
  }
  return 0;
}

cudaError_t launch_tree(int key_words, uint32_t used_bits, int grid, int threads, const ExploreArgs& args,
                        cudaStream_t stream) {
  void* params[] = {const_cast<ExploreArgs*>(&args)};
  return cudaLaunchCooperativeKernel(pick_tree(key_words, used_bits, args.prune != 0), dim3(grid), dim3(threads), params,
                                     0, stream);
}

}  // namespace mc
