// sf_stream.cuh - shared by the streaming passes (sf_stream.cu and the
// sf_tiled_*.cu translation units): the passes' parameters, the per-step
// epilogues, the row reductions, and how a launch is made.
#pragma once

#include <algorithm>
#include <array>
#include <numeric>
#include <type_traits>

#include "sf_device.cuh"
#include "sf_launch.h"

namespace sf {

// Kinds of pass: frontier (+ window aggregation), evidence, evidence with the
// telemetry-quality sums, routing baselines.
enum PassKind { kFrontier, kGain, kGainQuality, kBase };
__host__ __device__ constexpr bool is_gain(int kind) { return kind == kGain || kind == kGainQuality; }

constexpr int kRowBytes = 128;  // TMA row: 16 int64
constexpr int kRingBytes = 192 * 1024;
constexpr int kGainBytes = 213 * 1024;  // the evidence pass's ring and its windows' medians
constexpr int kMaxBoxRows = 256;  // the TMA box limit
constexpr int kMaxStages = 32;

// Consumer warps of a tiled pass.  The evidence pass does twice the work per
// byte (a median beside every duration) and is bound by the latency of its
// warps' chains, so it takes twelve, the most that leave 128 registers each,
// up to ten stages (six with the 128-bit quality sums); more need the registers
// (1024 x 10: 8 warps 1099 us, 12 warps 863 us).
__host__ __device__ constexpr int consumer_warps(int kind, int64_t S) {
  return (kind == kGain && S <= 10) || (kind == kGainQuality && S <= 6) ? 12 : 8;
}
// Small steps (regime 0): two ring stages per consumer warp.
__host__ __device__ constexpr int r0_stage_bytes(int kind, int64_t S) { return kRingBytes / (2 * consumer_warps(kind, S)); }
static_assert(r0_stage_bytes(kGain, 1) % 1024 == 0 && 2 * consumer_warps(kGain, 1) <= kMaxStages, "swizzled stages");

struct Params {
  int64_t T, R, S;
  // tiled path (launch_stream_pass): d and m seen as 128-byte rows of 16 int64
  int regime;         // 0: tiles of K whole steps, one warp each; 1: steps of tiles_per_step tiles
  int box_rows;       // rows a tile's copy takes
  int K, tiles_per_step;
  int tile_ranks;     // regime 1: ranks per tile
  int64_t rows, m_rows;  // whole rows of d and of m; the elements past them are read with plain loads
  int64_t* a;
  int32_t* lead;
  int64_t* mk;
  int64_t* X;
  int64_t* D;
  int64_t* E;
  int32_t* C;
  uint8_t* step_lead;
  int64_t t0, W, w_first;
  const int64_t* m;
  const int64_t* wall;
  int other_stage;
  int64_t eta_num, eta_den;
  int64_t* Y;
  uint64_t* quality;
  uint32_t* status;
  // evidence pass, regime 1: the medians of the window(s) in use stay in m_slots
  // (1 or 2) shared-memory slots of m_bytes each, copied in m_boxes boxes of
  // m_box_rows rows; or (m_slots 0) they stream beside every tile of d
  // (m_by_tma).  Regime 0 reads them from global memory.
  int m_slots, m_bytes, m_boxes, m_box_rows;
  int ring_bytes;  // stages and slots
  int m_by_tma;
  int nst, stage_bytes;  // ring stages in use and their size
  int groups;            // regime 1: consumer warp groups, each taking every groups-th step
  // routing-baseline pass
  const int64_t* d;
  int64_t* bM;
  uint64_t* bSUM;
  int64_t* bSLOW;
  int64_t* bRANK0;
};

// The tiled pass of a kind, over steps that are whole 128-byte rows (aligned,
// S even) or not.  map_m: the medians of the evidence pass.
using TiledLaunch = cudaError_t(const CUtensorMap& map, const CUtensorMap& map_m, const Params& p, int grid,
                                cudaStream_t stream, bool pdl);
TiledLaunch launch_frontier_aligned, launch_frontier_unaligned, launch_gain_aligned, launch_gain_unaligned,
    launch_quality_aligned, launch_quality_unaligned, launch_base_aligned, launch_base_unaligned;
// one lane per (step, stage)
cudaError_t launch_step_lanes(int kind, const Params& p, cudaStream_t stream, bool pdl);
// several steps per warp instruction: lanes_groups is their number G, 0 where the shape takes one
int lanes_groups(int64_t R, int64_t S);
cudaError_t launch_lanes(int G, const CUtensorMap& map, const Params& p, int grid, cudaStream_t stream, bool pdl);
namespace {

__device__ __forceinline__ uint32_t hi32(int64_t v) {
  return static_cast<uint32_t>(static_cast<uint64_t>(v) >> 32);
}

// --------------------------------------------------------------------------
// Window index of step t, (t0 + t) / W - w_first, recomputed (one 64-bit
// division) only when t passes the end of the last window seen: every thread
// visits its steps in increasing order, so that happens once per window
// rather than once per step.
struct WinTrack {
  int64_t lo = 0, hi = 0, w = 0;  // steps [lo, hi) belong to window w
  __device__ __forceinline__ int64_t at(int64_t t, int64_t t0, int64_t W, int64_t w_first) {
    if (t >= hi) {
      w = (t0 + t) / W - w_first;
      lo = (w + w_first) * W - t0;
      hi = lo + W;
    }
    return w;
  }
};

// Window accumulators held by the warp that finalizes steps: lane s keeps the
// stage-s numerators, every lane the denominator.
struct WinAcc {
  int64_t cur = -1;
  int64_t x = 0, y = 0, dsum = 0;
  int64_t erow = 0;  // E / C index of (window cur, this lane's stage, rank 0)
  WinTrack wt;
};

__device__ __forceinline__ void flush_window(const Params& p, int S, WinAcc& acc, int lane) {
  if (acc.cur >= 0) {
    if (lane < S) {
      if (acc.x) atomicAdd(reinterpret_cast<unsigned long long*>(&p.X[acc.cur * S + lane]),
                           static_cast<unsigned long long>(acc.x));
      if (p.Y && acc.y)
        atomicAdd(reinterpret_cast<unsigned long long*>(&p.Y[acc.cur * S + lane]),
                  static_cast<unsigned long long>(acc.y));
    }
    if (lane == 0 && acc.dsum)
      atomicAdd(reinterpret_cast<unsigned long long*>(&p.D[acc.cur]),
                static_cast<unsigned long long>(acc.dsum));
  }
  acc.x = acc.y = acc.dsum = 0;
}

// Frontier epilogue for step t.  Lane s < S holds the packed key
// (F[t,s] << 16) | (65535 - lead[t,s]); the whole warp participates.
__device__ __forceinline__ void finalize_frontier(const Params& p, int S, int64_t t, uint64_t key,
                                                  int lane, WinAcc& acc) {
  const bool valid = lane < S;
  const int64_t F = valid ? static_cast<int64_t>(key >> 16) : 0;
  const int32_t ld = valid ? 65535 - static_cast<int32_t>(key & 0xffffu) : 0;
  int64_t Fprev = __shfl_up_sync(kFull, F, 1);
  if (lane == 0) Fprev = 0;  // F[t,-1] = 0
  const int64_t a = valid ? F - Fprev : 0;
  const int64_t mk = __shfl_sync(kFull, F, S - 1);
  if (valid) {
    if (p.a) p.a[t * S + lane] = a;
    if (p.lead) p.lead[t * S + lane] = ld;
  }
  if (lane == 0 && p.mk) p.mk[t] = mk;
  if (p.X) {
    const int64_t w = acc.wt.at(t, p.t0, p.W, p.w_first);
    if (w != acc.cur) {
      flush_window(p, S, acc, lane);
      acc.cur = w;
      acc.erow = (w * S + lane) * p.R;
    }
    acc.x += a;
    acc.dsum += mk;
    if (valid && ld >= 0 && ld < p.R) {  // always true for valid input; guards flagged input
      const int64_t idx = acc.erow + ld;
      if (p.E && a != 0)
        atomicAdd(reinterpret_cast<unsigned long long*>(&p.E[idx]), static_cast<unsigned long long>(a));
      if (p.C) atomicAdd(&p.C[idx], 1);
    }
    if (p.step_lead) {
      const uint64_t k2 = valid ? ((static_cast<uint64_t>(a) << 5) | static_cast<uint64_t>(31 - lane)) : 0;
      const uint64_t km = warp_max_u64(k2);
      if (lane == 0) p.step_lead[t] = static_cast<uint8_t>(31 - static_cast<int>(km & 31u));
    }
  }
}

// Evidence epilogue for step t.  Lane s < S holds the packed frontier key
// (F[t,s] << 16) | (65535 - lead[t,s]) and
// Fr[t,s] = max_r (P[t,r,S-1] - max(0, d[t,r,s] - m[w,r,s])).
// w: the step's window.
__device__ __forceinline__ void finalize_gain(const Params& p, int S, int64_t t, int64_t w, uint64_t key,
                                              int64_t Fr, int lane, WinAcc& acc) {
  const bool valid = lane < S;
  const int64_t F = valid ? static_cast<int64_t>(key >> 16) : 0;
  const int32_t ld = valid ? 65535 - static_cast<int32_t>(key & 0xffffu) : 0;
  int64_t Fprev = __shfl_up_sync(kFull, F, 1);
  if (lane == 0) Fprev = 0;
  const int64_t a = valid ? F - Fprev : 0;
  const int64_t FS = __shfl_sync(kFull, F, S - 1);
  const int64_t y = valid ? FS - Fr : 0;
  // leading stage (largest increment, lowest stage) and the runner-up increment
  const uint64_t k2 = valid ? ((static_cast<uint64_t>(a) << 5) | static_cast<uint64_t>(31 - lane)) : 0;
  const uint64_t km = warp_max_u64(k2);
  const int best = 31 - static_cast<int>(km & 31u);
  const int64_t amax = static_cast<int64_t>(km >> 5);
  const int64_t second = static_cast<int64_t>(warp_max_u64(valid && lane != best ? static_cast<uint64_t>(a) : 0));
  const bool conf = FS > 0 && static_cast<__int128>(amax - second) * p.eta_den >=
                                  static_cast<__int128>(p.eta_num) * FS;
  if (lane == 0) p.step_lead[t] = static_cast<uint8_t>(best | (conf ? SF_STEP_CONFIDENT : 0u));
  if (w != acc.cur) {
    flush_window(p, S, acc, lane);
    acc.cur = w;
    acc.erow = (w * S + lane) * p.R;
  }
  acc.x += a;
  acc.y += y;
  acc.dsum += FS;
  if (valid && ld >= 0 && ld < p.R) {  // lead-rank credit (always in range for valid input)
    const int64_t idx = acc.erow + ld;
    if (p.E && a != 0)
      atomicAdd(reinterpret_cast<unsigned long long*>(&p.E[idx]), static_cast<unsigned long long>(a));
    if (p.C) atomicAdd(&p.C[idx], 1);
  }
}

// Routing-baseline window accumulators (lane s: stage s).
struct BaseAcc {
  int64_t cur = -1;
  int64_t m = 0, slow = 0, r0 = 0;
  unsigned __int128 sum = 0;
  WinTrack wt;
};

__device__ __forceinline__ void flush_base(const Params& p, int S, BaseAcc& acc, int lane) {
  if (acc.cur >= 0 && lane < S) {
    const int64_t i = acc.cur * S + lane;
    if (acc.m) atomicAdd(reinterpret_cast<unsigned long long*>(&p.bM[i]), static_cast<unsigned long long>(acc.m));
    if (acc.sum) atomic_add_u128(p.bSUM + 2 * i, acc.sum);
    if (acc.slow)
      atomicAdd(reinterpret_cast<unsigned long long*>(&p.bSLOW[i]), static_cast<unsigned long long>(acc.slow));
    if (acc.r0) atomicAdd(reinterpret_cast<unsigned long long*>(&p.bRANK0[i]), static_cast<unsigned long long>(acc.r0));
  }
  acc.m = acc.slow = acc.r0 = 0;
  acc.sum = 0;
}

// Baseline epilogue for step t.  Lane s < S holds max_r d[t,r,s] and
// sum_r d[t,r,s]; every lane holds the packed key of the slowest rank
// (largest total, lowest rank on ties), whose row and rank 0's row are read
// back from d (the step was just streamed, so these hit L2).
__device__ __forceinline__ void finalize_base(const Params& p, int S, int64_t t, uint64_t mx, uint64_t sm,
                                              uint64_t slowkey, int lane, BaseAcc& acc) {
  const int64_t w = acc.wt.at(t, p.t0, p.W, p.w_first);
  if (w != acc.cur) {
    flush_base(p, S, acc, lane);
    acc.cur = w;
  }
  const int64_t rs = 65535 - static_cast<int64_t>(slowkey & 0xffffu);
  if (lane < S && rs >= 0 && rs < p.R) {  // always in range for valid input
    acc.m += static_cast<int64_t>(mx);
    acc.sum += sm;
    acc.slow += __ldg(p.d + (t * p.R + rs) * S + lane);
    acc.r0 += __ldg(p.d + t * p.R * S + lane);
  }
}

// Three 32-bit sums of 24-, 24- and 16-bit parts (no carry can be lost in them).
__device__ __forceinline__ uint64_t warp_sum_u64(uint64_t v) {
  const uint32_t a = __reduce_add_sync(kFull, static_cast<uint32_t>(v) & 0xffffffu);
  const uint32_t b = __reduce_add_sync(kFull, static_cast<uint32_t>(v >> 24) & 0xffffffu);
  const uint32_t c = __reduce_add_sync(kFull, static_cast<uint32_t>(v >> 48));
  return a + (static_cast<uint64_t>(b) << 24) + (static_cast<uint64_t>(c) << 48);
}

// Telemetry-quality sums of one thread (App. A closure / overlap), flushed per window.
struct QualAcc {
  int64_t cur = -1;
  unsigned __int128 res = 0, ovl = 0, wsum = 0;
};

__device__ __forceinline__ unsigned __int128 warp_sum_u128(unsigned __int128 v) {
  uint64_t lo = static_cast<uint64_t>(v), hi = static_cast<uint64_t>(v >> 64);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const uint64_t olo = __shfl_xor_sync(kFull, lo, o);
    const uint64_t ohi = __shfl_xor_sync(kFull, hi, o);
    const uint64_t nlo = lo + olo;
    hi = hi + ohi + (nlo < lo ? 1u : 0u);
    lo = nlo;
  }
  return (static_cast<unsigned __int128>(hi) << 64) | lo;
}

// Warp-uniform: every lane calls with the same window index w.
__device__ __forceinline__ void qual_window(const Params& p, QualAcc& q, int64_t w, int lane) {
  if (w == q.cur) return;
  if (q.cur >= 0) {
    const unsigned __int128 r = warp_sum_u128(q.res), o = warp_sum_u128(q.ovl), s = warp_sum_u128(q.wsum);
    if (lane == 0) {
      uint64_t* dst = p.quality + q.cur * 6;
      if (r) atomic_add_u128(dst + 0, r);
      if (o) atomic_add_u128(dst + 2, o);
      if (s) atomic_add_u128(dst + 4, s);
    }
  }
  q.res = q.ovl = q.wsum = 0;
  q.cur = w;
}

__device__ __forceinline__ void qual_row(const Params& p, QualAcc& q, int64_t t, int64_t r,
                                         int64_t total, int64_t other, uint32_t& dor) {
  if (p.wall) {
    const int64_t wv = p.wall[t * p.R + r];
    dor |= hi32(wv);
    const int64_t e = wv - (total - other);  // e = w - sum_{s != other} d
    if (e > 0) q.res += static_cast<uint64_t>(e);
    else q.ovl += static_cast<uint64_t>(-e);
    q.wsum += static_cast<uint64_t>(wv);
  } else {
    q.res += static_cast<uint64_t>(other);
    q.wsum += static_cast<uint64_t>(total);
  }
}

// --------------------------------------------------------------------------
// Per-thread running maxima over the rank rows a thread visits (in increasing
// rank order, so a strict '>' keeps the lowest rank on ties).
template <int S>
struct FrontierRows {
  int64_t bp[S];
  int32_t br[S];
  __device__ __forceinline__ void init() {
#pragma unroll
    for (int s = 0; s < S; ++s) {
      bp[s] = -1;
      br[s] = 0;
    }
  }
  __device__ __forceinline__ void row(const int64_t (&v)[S], int32_t r, uint32_t& dor, uint32_t& tor) {
    int64_t P = 0;
#pragma unroll
    for (int s = 0; s < S; ++s) {
      dor |= hi32(v[s]);
      P += v[s];  // P[t,r,s]
      if (P > bp[s]) {
        bp[s] = P;
        br[s] = r;
      }
    }
    tor |= hi32(P);
  }
  __device__ __forceinline__ uint64_t key(int s) const {
    return bp[s] < 0 ? 0ull
                     : (static_cast<uint64_t>(bp[s]) << 16) | static_cast<uint64_t>(65535 - br[s]);
  }
};

__host__ __device__ constexpr int ceil_log2(int x) { return x <= 1 ? 0 : 1 + ceil_log2((x + 1) / 2); }

// Evidence-pass maxima, with the frontier's lowest attaining rank.  A row is
// narrow when its durations and medians are below 2^32 ns and its total below
// 2^32 - 1 ns (4.29 s a step): every prefix then fits 32 bits, and so does
// P_S - (max(d, m) - m), which is P_S - max(0, d - m).  A thread keeps 32-bit
// maxima until it meets the first other row (a long step, invalid input);
// from there on its step runs in 64 bits, in the same registers: the words
// that held a prefix and its rank hold the packed key (F << 16) | (65535 - r).
// A thread that met such a row starts its next step in 64 bits.  Rows arrive in increasing rank order, so a strict '>' keeps the lowest rank
// on ties.
template <int S>
struct GainRows {
  static constexpr int kPairs = (S + 1) / 2;
  uint32_t a[S], b[S];   // narrow: 1 + max_r P[t,r,s] (0: none) and the lowest rank attaining it; wide: key, high and low word
  uint32_t g[S], gh[S];  // max_r (P_S - max(0, d - m)), low and high word
  bool wide;             // the state is 64-bit
  bool met;              // a row of this step was not narrow
  __device__ __forceinline__ void init(bool start_wide) {
#pragma unroll
    for (int s = 0; s < S; ++s) a[s] = b[s] = g[s] = gh[s] = 0;
    wide = start_wide;
    met = false;
  }
  __device__ __forceinline__ uint64_t key(int s) const {
    if (wide) return (static_cast<uint64_t>(a[s]) << 32) | b[s];
    return a[s] ? (static_cast<uint64_t>(a[s] - 1) << 16) | static_cast<uint64_t>(65535u - b[s]) : 0ull;
  }
  __device__ __forceinline__ uint64_t gain(int s) const { return (static_cast<uint64_t>(gh[s]) << 32) | g[s]; }

  // dp(j) and mp(j): stages 2j and 2j + 1 of the row and of its medians (0 past
  // the last stage).  Only low words are held; a wide row is read again.
  template <typename DPair, typename MPair>
  __device__ __forceinline__ int64_t row(DPair dp, MPair mp, int32_t r, uint32_t& dor, uint32_t& tor) {
    if (!wide) {
      uint32_t x[S], y[S];
      uint32_t big = 0;
      uint64_t total = 0;
#pragma unroll
      for (int j = 0; j < kPairs; ++j) {
        const longlong2 u = dp(j), m = mp(j);
        x[2 * j] = static_cast<uint32_t>(u.x);
        y[2 * j] = static_cast<uint32_t>(m.x);
        if (2 * j + 1 < S) {
          x[2 * j + 1] = static_cast<uint32_t>(u.y);
          y[2 * j + 1] = static_cast<uint32_t>(m.y);
        }
        big |= hi32(u.x) | hi32(u.y) | hi32(m.x) | hi32(m.y);
        total += static_cast<uint64_t>(static_cast<uint32_t>(u.x)) + static_cast<uint32_t>(u.y);
      }
      // no duration has a high word, so the prefixes do not decrease and the total bounds them
      big |= static_cast<uint32_t>((total + 1) >> 32);
      if (big == 0) {
        const uint32_t Pt = static_cast<uint32_t>(total);
        uint32_t P1 = 1;
#pragma unroll
        for (int s = 0; s < S; ++s) {
          P1 += x[s];
          b[s] = P1 > a[s] ? static_cast<uint32_t>(r) : b[s];
          a[s] = max(P1, a[s]);
          g[s] = max(g[s], Pt - max(x[s], y[s]) + y[s]);
        }
        return static_cast<int64_t>(Pt);
      }
    }
    if (!wide) {  // the first such row: the maxima so far become keys
#pragma unroll
      for (int s = 0; s < S; ++s) {
        const uint64_t k = key(s);
        a[s] = static_cast<uint32_t>(k >> 32);
        b[s] = static_cast<uint32_t>(k);
      }
      wide = true;
    }
    return row_wide(dp, mp, r, dor, tor);
  }

  template <typename DPair, typename MPair>
  __device__ __forceinline__ int64_t row_wide(DPair dp, MPair mp, int32_t r, uint32_t& dor, uint32_t& tor) {
    asm volatile("" ::: "memory");  // the row is read again, not kept in registers by its caller
    int64_t P = 0;
    uint32_t big = 0;
#pragma unroll
    for (int j = 0; j < kPairs; ++j) {
      const longlong2 u = dp(j);
      big |= hi32(u.x) | hi32(u.y);
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int s = 2 * j + h;
        if (s >= S) break;
        P += h ? u.y : u.x;
        const uint64_t k = (static_cast<uint64_t>(P) << 16) | static_cast<uint64_t>(65535 - r);
        const uint64_t old = (static_cast<uint64_t>(a[s]) << 32) | b[s];
        const uint64_t best = k > old ? k : old;
        a[s] = static_cast<uint32_t>(best >> 32);
        b[s] = static_cast<uint32_t>(best);
      }
    }
    dor |= big;
    tor |= hi32(P);
    big |= hi32(P + 1);
    if constexpr (S > 8) asm volatile("" ::: "memory");
#pragma unroll
    for (int j = 0; j < kPairs; ++j) {
      const longlong2 u = dp(j), m = mp(j);
      big |= hi32(m.x) | hi32(m.y);
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int s = 2 * j + h;
        if (s >= S) break;
        const int64_t v = h ? u.y : u.x, mv = h ? m.y : m.x;
        const int64_t alt = P - (v > mv ? v - mv : 0), old = static_cast<int64_t>(gain(s));
        const uint64_t best = static_cast<uint64_t>(alt > old ? alt : old);
        g[s] = static_cast<uint32_t>(best);
        gh[s] = static_cast<uint32_t>(best >> 32);
      }
    }
    met |= big != 0;
    return P;
  }

  // The warp's maxima of stage s: k = (F << 16) | (65535 - lead), 0 when no
  // lane saw a row; `narrow`: no lane is wide.
  __device__ __forceinline__ void warp_max(int s, bool narrow, uint64_t& k, uint64_t& G) const {
    if (narrow) {
      const uint32_t m = __reduce_max_sync(kFull, a[s]);
      const uint32_t lead = __reduce_min_sync(kFull, a[s] == m ? b[s] : 0xffffffffu);
      k = m ? (static_cast<uint64_t>(m - 1) << 16) | static_cast<uint64_t>(65535u - lead) : 0ull;
      G = __reduce_max_sync(kFull, g[s]);
    } else {
      k = warp_max_u64(key(s));
      G = warp_max_u64(gain(s));
    }
  }
};

// Routing-baseline maxima and sums over the rank rows a thread visits.
template <int S>
struct BaseRows {
  int64_t mx[S];
  uint64_t sm[S];
  uint64_t slow;  // (P_S << 16) | (65535 - r), max
  __device__ __forceinline__ void init() {
#pragma unroll
    for (int s = 0; s < S; ++s) {
      mx[s] = 0;
      sm[s] = 0;
    }
    slow = 0;
  }
  __device__ __forceinline__ void row(const int64_t (&v)[S], int32_t r, uint32_t& dor, uint32_t& tor) {
    int64_t P = 0;
#pragma unroll
    for (int s = 0; s < S; ++s) {
      dor |= hi32(v[s]);
      P += v[s];
      mx[s] = v[s] > mx[s] ? v[s] : mx[s];
      sm[s] += static_cast<uint64_t>(v[s]);
    }
    tor |= hi32(P);
    const uint64_t k = (static_cast<uint64_t>(P) << 16) | static_cast<uint64_t>(65535 - r);
    slow = k > slow ? k : slow;
  }
};


// Launch `kern` on `stream`; with `pdl`, as the programmatic dependent of the
// previous launch on the stream (this call's clear of its outputs: the kernel
// streams its first tiles while the clear runs and writes after griddep_wait).
template <typename... KArgs, typename... Args>
cudaError_t launch_ex(void (*kern)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t stream, bool pdl,
                      Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = pdl ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kern, args...);
}

}  // namespace
}  // namespace sf
