// sf_tiled.cuh - the tiled streaming pass, instantiated per kind of pass by
// the sf_tiled_*.cu files.
//
// A persistent grid, one CTA per SM, each CTA owning a contiguous range of
// steps.  Producer threads stream 128-byte rows of d into a ring of
// shared-memory tiles with 2-D bulk tensor copies (TMA) completing on
// mbarriers; the consumer warps read whole rank rows out of the tiles, keep
// the prefix and per-boundary maxima in registers, and reduce across ranks
// with warp redux plus one shared-memory exchange.
//
// Any rank count and up to 16 stages: a tile starts at the 128-byte row that
// holds its first element, and rank rows are read at that element's offset in
// the row (with R*S a multiple of 16 and S even, 0 in every tile: the ALIGNED
// kernels, whose swizzled addresses need no arithmetic per load).  Elements past
// the last whole row of d are written into the tile by its readers.  Steps that
// are not whole rows took a warp or a CTA each with plain loads before: evidence
// pass over 4001 x 1001 x 13 572 -> 105 us, 13421 x 1000 x 5 279 -> 129 us.  The tiles are
// 128B-swizzled for 4, 8 and 16 stages, where the 16-byte reads of consecutive
// rank rows would share banks; for other even and for odd stage counts the
// rows' stride already spreads them.
#pragma once

#include "sf_median_slots.h"
#include "sf_stream.cuh"

namespace sf {
namespace {

constexpr int kProducers = 4;    // producer warps: no cost in registers, which go by warps in fours
constexpr int kRedPerWarp = 64;  // per-warp partials of one step (<= 2S + 1)
constexpr size_t tiled_smem(int kind, int64_t S, int ring) {
  return 1024 /*alignment slack*/ + size_t(ring) + (2 * kMaxStages + 4) * sizeof(uint64_t) + 16 +
         size_t(2) * consumer_warps(kind, S) * kRedPerWarp * sizeof(uint64_t);  // partials double-buffered
}
static_assert(tiled_smem(kGain, 1, kGainBytes) <= 227 * 1024, "shared memory of one CTA");

// The place of element e of a tile, and 16-byte chunk c.
template <bool kSwz>
__device__ __forceinline__ int chunk_at(int c) {
  return (kSwz ? (c ^ ((c >> 3) & 7)) : c) * 16;
}

// Stages 2j and 2j + 1 (0 past the last stage) of the tile's rank row q, the
// tile's first rank row starting at element `off`.
template <int S, bool kSwz>
__device__ __forceinline__ longlong2 tile_pair(const unsigned char* tile, int off, int q, int j) {
  if constexpr (S % 2 == 0) {
    return *reinterpret_cast<const longlong2*>(tile + chunk_at<kSwz>((off >> 1) + q * (S / 2) + j));
  } else {
    const int64_t* at = reinterpret_cast<const int64_t*>(tile) + off + q * S + 2 * j;
    return make_longlong2(at[0], 2 * j + 1 < S ? at[1] : 0);
  }
}

// Stage `idx` of the row, 0 for idx < 0.
template <int S, bool kSwz>
__device__ __forceinline__ int64_t tile_stage(const unsigned char* tile, int off, int q, int idx) {
  if (idx < 0) return 0;
  const int e = off + q * S + idx;
  return *reinterpret_cast<const int64_t*>(tile + chunk_at<kSwz>(e >> 1) + (e & 1) * 8);
}

template <int S, bool kSwz>
__device__ __forceinline__ void load_row(const unsigned char* tile, int off, int q, int64_t (&v)[S]) {
#pragma unroll
  for (int j = 0; j < (S + 1) / 2; ++j) {
    const longlong2 x = tile_pair<S, kSwz>(tile, off, q, j);
    v[2 * j] = x.x;
    if (2 * j + 1 < S) v[2 * j + 1] = x.y;
  }
}

// Elements [rows * 16, first + n) of the tensor `src`, past its whole rows,
// written to their places in the tile that starts at the row of element
// `first`.  Every warp that reads the tile calls it (the same values land).
template <bool kSwz>
__device__ __forceinline__ void patch_tail(unsigned char* tile, const int64_t* src, int64_t rows, int64_t first, int n,
                                           int lane) {
  const int64_t e0 = first & ~int64_t(15), end = first + n;
  if (end <= rows * 16) return;
  for (int64_t e = rows * 16 + lane; e < end; e += 32) {
    const int at = static_cast<int>(e - e0);
    *reinterpret_cast<int64_t*>(tile + chunk_at<kSwz>(at >> 1) + (at & 1) * 8) = __ldg(src + e);
  }
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // before a later copy into this stage
  __syncwarp();
}

// Ring stage and phase parity of the j-th tile a CTA streams.
// Regime 0: tile j belongs to warp j % W, which alternates its two stages.
template <int W>
__device__ __forceinline__ void stage_of_r0(uint32_t j, uint32_t& st, uint32_t& ph) {
  const uint32_t i = j / W;
  st = 2u * (j % W) + (i & 1u);
  ph = (i >> 1) & 1u;
}

// Regime 1: the steps go to the warp groups in turn; group g owns stages g,
// g + G, ..., g + G (nst / G - 1) and fills them in that order.  The walk of
// one group's stages, kept incrementally (no division per tile).
struct GroupRing {
  uint32_t slot = 0, ph = 0;  // next stage slot within the group and its phase parity
  __device__ __forceinline__ uint32_t stage(uint32_t g, uint32_t G) const { return g + G * slot; }
  __device__ __forceinline__ void advance(uint32_t spg) {
    if (++slot == spg) {
      slot = 0;
      ph ^= 1u;
    }
  }
};


// Window slots of resident medians (sf_median_slots.h) and their barriers.
struct MedianSlots {
  unsigned char* base;
  uint64_t *full, *done;  // [2] each
};

// Producer q of kProducers (one thread each) issues the copies of the stages
// that belong to it: regime 0, those of the warps q, q + 4, ...; regime 1, those
// of warp group q (with one group, all by producer 0).  A step's wait for its
// own group's stages then holds up no other group's copies (evidence pass, one
// producer in step order against four: 1024 x 10 809 / 751 us, 300 x 10 217 /
// 174 us, 2000 x 8 280 / 230 us).
template <int W>
__device__ void produce(int q, const CUtensorMap* map, const CUtensorMap* map_m, const Params& p, int64_t t_begin,
                        int64_t t_end, unsigned char* ring, uint64_t* full, uint64_t* empty, const MedianSlots& ms,
                        volatile int* abort) {
  static_assert(W % kProducers == 0, "each consumer warp's stages belong to one producer");
  const uint32_t G = static_cast<uint32_t>(p.groups);
  if (p.regime == 1 && q >= p.groups) return;
  prefetch_tensormap(map);
  if (p.m_by_tma || p.m_slots) prefetch_tensormap(map_m);
  const uint32_t bytes = static_cast<uint32_t>(p.box_rows) * kRowBytes;
  const int64_t RS = p.R * p.S;
  uint32_t used = 0, last_ph = 0;  // per stage: issued into at all, parity of the last issue
  bool ok = true;
  auto issue = [&](int64_t row, int64_t mrow, uint32_t st, uint32_t ph) {
    if (!mbar_wait_bounded(&empty[st], ph ^ 1u, abort)) {
      ok = false;
      return;
    }
    used |= 1u << st;
    last_ph = (last_ph & ~(1u << st)) | (ph << st);
    unsigned char* dst = ring + size_t(st) * p.stage_bytes;
    mbar_arrive_expect_tx(&full[st], p.m_by_tma ? 2u * bytes : bytes);
    tma_load_2d(dst, map, 0, static_cast<int32_t>(row), &full[st]);
    if (p.m_by_tma) tma_load_2d(dst + p.stage_bytes / 2, map_m, 0, static_cast<int32_t>(mrow), &full[st]);
  };
  WinTrack mw;  // window of the medians (evidence pass)
  int m_next = 0;  // windows of resident medians issued
  const MedianPlace place{p.m_slots};
  const int64_t w_base = p.m_slots ? t_begin / p.W : 0;
  // producer 0: the resident medians of every window up to that of step t
  auto medians_to = [&](int64_t t) {
    if (q != 0 || !p.m_slots) return;
    for (const int last = static_cast<int>(mw.at(t, 0, p.W, 0) - w_base); m_next <= last && ok; ++m_next) {
      const uint32_t sl = place.slot(m_next);
      if (!mbar_wait_bounded(&ms.done[sl], place.parity(m_next) ^ 1u, abort)) {
        ok = false;
        return;
      }
      mbar_arrive_expect_tx(&ms.full[sl], static_cast<uint32_t>(p.m_bytes));
      const int64_t row = ((m_next + w_base) * RS) >> 4;
      for (int b = 0; b < p.m_boxes; ++b)
        tma_load_2d(ms.base + size_t(sl) * p.m_bytes + size_t(b) * p.m_box_rows * kRowBytes, map_m, 0,
                    static_cast<int32_t>(row + int64_t(b) * p.m_box_rows), &ms.full[sl]);
    }
  };
  if (p.regime == 0) {
    uint32_t j = static_cast<uint32_t>(q);
    for (int64_t t = t_begin + int64_t(q) * p.K; t < t_end && ok; t += int64_t(kProducers) * p.K, j += kProducers) {
      uint32_t st, ph;
      stage_of_r0<W>(j, st, ph);
      issue((t * RS) >> 4, 0, st, ph);
    }
  } else {
    const uint32_t spg = static_cast<uint32_t>(p.nst) / G;
    uint32_t slot = 0, ph = 0;
    for (int64_t t = t_begin + q; t < t_end && ok; t += G) {
      medians_to(t);
      const int64_t mrow = p.m_by_tma ? mw.at(t, 0, p.W, 0) * RS : 0;
      for (int k = 0; k < p.tiles_per_step && ok; ++k) {
        const int64_t e0 = min(int64_t(k) * p.tile_ranks, p.R - p.tile_ranks) * p.S;
        issue((t * RS + e0) >> 4, (mrow + e0) >> 4, static_cast<uint32_t>(q) + G * slot, ph);
        if (++slot == spg) {
          slot = 0;
          ph ^= 1u;
        }
      }
      // a window that starts at the other groups' steps of this round: only now,
      // since this group's step may be the last that its slot waits for
      medians_to(min(t + G, t_end) - 1);
    }
  }
  // copies still in flight: at most one per stage and slot, the last issued into it
  for (uint32_t st = 0; st < kMaxStages; ++st)
    if ((used >> st) & 1u) mbar_wait_timeout(&full[st], (last_ph >> st) & 1u);
  for (int i = max(0, m_next - p.m_slots); i < m_next; ++i)
    mbar_wait_timeout(&ms.full[place.slot(i)], place.parity(i));
}

// --------------------------------------------------------------------------
template <int S, int KIND, bool ALIGNED>
__global__ void __launch_bounds__((consumer_warps(KIND, S) + kProducers) * 32, 1)
    stream_kernel(const __grid_constant__ CUtensorMap map, const __grid_constant__ CUtensorMap map_m,
                  const Params p) {
  constexpr bool GAIN = is_gain(KIND);
  constexpr bool QUALITY = KIND == kGainQuality;
  constexpr bool BASE = KIND == kBase;
  constexpr int kWarps = consumer_warps(KIND, S);
  constexpr bool kSwz = (S == 4 || S == 8 || S == 16);
  constexpr int U = S <= 8 ? 4 : 2;  // rank rows in flight per thread
  extern __shared__ unsigned char smem_raw[];
  unsigned char* ring = align_1024(smem_raw);
  uint64_t* full = reinterpret_cast<uint64_t*>(ring + p.ring_bytes);
  uint64_t* empty = full + kMaxStages;
  volatile int* abort = reinterpret_cast<volatile int*>(empty + kMaxStages);
  uint64_t* red = reinterpret_cast<uint64_t*>(empty + kMaxStages) + 6;
  // resident medians: after the ring's stages; their barriers after the abort word
  const MedianSlots ms = {ring + size_t(p.nst) * p.stage_bytes, empty + kMaxStages + 2, empty + kMaxStages + 4};

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t G = gridDim.x, b = blockIdx.x;
  const int64_t t_begin = p.T * b / G, t_end = p.T * (b + 1) / G;

  if (threadIdx.x < kMaxStages) {
    mbar_init(&full[threadIdx.x], 1);
    mbar_init(&empty[threadIdx.x], p.regime == 0 ? 1u : uint32_t(kWarps / p.groups));
    if (threadIdx.x < 2) {
      mbar_init(&ms.full[threadIdx.x], 1);
      mbar_init(&ms.done[threadIdx.x], uint32_t(kWarps));
    }
    if (threadIdx.x == 0) *abort = 0;
    fence_barrier_init();
  }
  __syncthreads();

  if (warp >= kWarps) {
    if (lane == 0) produce<kWarps>(warp - kWarps, &map, &map_m, p, t_begin, t_end, ring, full, empty, ms, abort);
    return;
  }
  griddep_wait();  // outputs cleared by the launch before this one (when it is its dependent)

  uint32_t dor = 0, tor = 0;  // OR of duration / rank-total high words
  WinAcc acc;
  QualAcc qa;
  WinTrack qt;  // window of the step a warp is on (evidence pass)
  BaseAcc bacc;
  [[maybe_unused]] bool start_wide = false;  // evidence: this thread's last step held a row past 32 bits
  const int R = static_cast<int>(p.R);
  const int64_t RS = p.R * S;
  // resident medians of a step's window: the slot, once they have landed
  [[maybe_unused]] MedianWalk mwalk;
  [[maybe_unused]] const MedianPlace place{p.m_slots};
  [[maybe_unused]] const int64_t w_base = GAIN && p.m_slots ? t_begin / p.W : 0;
  [[maybe_unused]] bool m_have = true;
  auto hand_back = [&](int i) {
    if (lane == 0) mbar_arrive(&ms.done[place.slot(i)]);
  };
  auto landed = [&](int i) {
    if (!mbar_wait_bounded(&ms.full[place.slot(i)], place.parity(i), abort)) m_have = false;
  };
  auto enter = [&](int64_t w) {
    const int i = static_cast<int>(w - w_base);
    if (mwalk.at == i) return;
    __syncwarp();  // every lane's reads of the window left behind are done
    mwalk.enter(i, hand_back, landed);
    if (!ALIGNED && m_have)
      patch_tail<kSwz>(ms.base + size_t(place.slot(i)) * p.m_bytes, p.m, p.m_rows, w * RS, static_cast<int>(RS), lane);
  };

  if (p.regime == 0) {
    // ---- the warps take the tiles (K whole steps) in turn, each with two ring stages
    const int64_t n_local = t_end - t_begin;
    const int64_t n_tiles = (n_local + p.K - 1) / p.K;
    uint32_t i = 0;
    for (int64_t j = warp; j < n_tiles; j += kWarps, ++i) {
      const uint32_t st = 2u * warp + (i & 1u), ph = (i >> 1) & 1u;
      const bool have = mbar_wait_bounded(&full[st], ph, abort);
      unsigned char* tile = ring + size_t(st) * r0_stage_bytes(KIND, S);
      const int nsteps = static_cast<int>(min(int64_t(p.K), n_local - j * p.K));
      const int64_t first = (t_begin + j * p.K) * RS;  // the tile's first element
      const int off = ALIGNED ? 0 : static_cast<int>(first & 15);
      if (!ALIGNED && have) patch_tail<kSwz>(tile, p.d, p.rows, first, nsteps * static_cast<int>(RS), lane);
      int kk0 = 0;
      if constexpr (KIND == kFrontier && S <= 8) {
        // frontier steps in pairs: two independent reduction chains per warp
        constexpr int UP = S <= 4 ? 2 : 1;  // rank rows of each step in flight per lane
        for (; kk0 + 1 < nsteps; kk0 += 2) {
          const int64_t t = t_begin + j * p.K + kk0;
          FrontierRows<S> ra, rb;
          ra.init();
          rb.init();
          if (have) {
            for (int r0 = lane; r0 < R; r0 += 32 * UP) {
              int64_t va[UP][S], vb[UP][S];
#pragma unroll
              for (int u = 0; u < UP; ++u)
                if (r0 + 32 * u < R) {
                  load_row<S, kSwz>(tile, off, kk0 * R + r0 + 32 * u, va[u]);
                  load_row<S, kSwz>(tile, off, (kk0 + 1) * R + r0 + 32 * u, vb[u]);
                }
#pragma unroll
              for (int u = 0; u < UP; ++u)
                if (r0 + 32 * u < R) {
                  ra.row(va[u], r0 + 32 * u, dor, tor);
                  rb.row(vb[u], r0 + 32 * u, dor, tor);
                }
            }
          }
          uint64_t ka = 0, kb = 0;
#pragma unroll
          for (int s = 0; s < S; ++s) {
            const uint64_t ma = warp_max_u64(ra.key(s));
            const uint64_t mb = warp_max_u64(rb.key(s));
            if (lane == s) {
              ka = ma;
              kb = mb;
            }
          }
          finalize_frontier(p, S, t, ka, lane, acc);
          finalize_frontier(p, S, t + 1, kb, lane, acc);
        }
      }
      for (int kk = kk0; kk < nsteps; ++kk) {
        const int64_t t = t_begin + j * p.K + kk;
        const int64_t w = GAIN ? qt.at(t, 0, p.W, 0) : 0;
        if (QUALITY) qual_window(p, qa, w, lane);
        const int q0 = kk * R;
        if constexpr (KIND == kFrontier) {
          FrontierRows<S> rs;
          rs.init();
          if (have) {
            for (int r0 = lane; r0 < R; r0 += 32 * U) {
              int64_t v[U][S];
#pragma unroll
              for (int u = 0; u < U; ++u)
                if (r0 + 32 * u < R) load_row<S, kSwz>(tile, off, q0 + r0 + 32 * u, v[u]);
#pragma unroll
              for (int u = 0; u < U; ++u)
                if (r0 + 32 * u < R) rs.row(v[u], r0 + 32 * u, dor, tor);
            }
          }
          uint64_t mykey = 0;
#pragma unroll
          for (int s = 0; s < S; ++s) {
            const uint64_t km = warp_max_u64(rs.key(s));
            if (lane == s) mykey = km;
          }
          finalize_frontier(p, S, t, mykey, lane, acc);
        } else if constexpr (BASE) {
          BaseRows<S> rs;
          rs.init();
          if (have) {
            for (int r0 = lane; r0 < R; r0 += 32 * U) {
              int64_t v[U][S];
#pragma unroll
              for (int u = 0; u < U; ++u)
                if (r0 + 32 * u < R) load_row<S, kSwz>(tile, off, q0 + r0 + 32 * u, v[u]);
#pragma unroll
              for (int u = 0; u < U; ++u)
                if (r0 + 32 * u < R) rs.row(v[u], r0 + 32 * u, dor, tor);
            }
          }
          uint64_t myM = 0, mySum = 0;
#pragma unroll
          for (int s = 0; s < S; ++s) {
            const uint64_t mx = warp_max_u64(static_cast<uint64_t>(rs.mx[s]));
            const uint64_t sm = warp_sum_u64(rs.sm[s]);
            if (lane == s) {
              myM = mx;
              mySum = sm;
            }
          }
          finalize_base(p, S, t, myM, mySum, warp_max_u64(rs.slow), lane, bacc);
        } else {
          GainRows<S> rs;
          rs.init(start_wide);
          if (have) {
            for (int r = lane; r < R; r += 32) {
              const int64_t* mrow = p.m + (w * p.R + r) * S;
              auto median_pair = [&](int h) -> longlong2 {
                if constexpr (S % 2 == 0) return __ldg(reinterpret_cast<const longlong2*>(mrow) + h);
                else return make_longlong2(__ldg(mrow + 2 * h), 2 * h + 1 < S ? __ldg(mrow + 2 * h + 1) : 0);
              };
              const int64_t total = rs.row([&](int h) { return tile_pair<S, kSwz>(tile, off, q0 + r, h); },
                                           median_pair, r, dor, tor);
              if constexpr (QUALITY)
                qual_row(p, qa, t, r, total, tile_stage<S, kSwz>(tile, off, q0 + r, p.other_stage), dor);
            }
          }
          uint64_t myK = 0;
          int64_t myR = 0;
          const bool narrow = !__any_sync(kFull, rs.wide);
          start_wide = rs.met;
#pragma unroll
          for (int s = 0; s < S; ++s) {
            uint64_t f, g;
            rs.warp_max(s, narrow, f, g);
            if (lane == s) {
              myK = f;
              myR = static_cast<int64_t>(g);
            }
          }
          finalize_gain(p, S, t, w, myK, myR, lane, acc);
        }
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(&empty[st]);
    }
  } else {
    // ---- one step per warp group (of kWarps / groups warps), the
    // groups taking steps in turn, tiles_per_step tiles per step
    // (the group count is a compile-time constant in each copy of the loop)
    auto consume = [&](auto ng) {
      constexpr int NG = decltype(ng)::value;
      constexpr int gw = kWarps / NG;  // warps per group
      const int g = warp / gw, lw = warp % gw;
      constexpr int gthreads = gw * 32;
      const int ctid = threadIdx.x - g * gthreads;  // thread within the group
      const uint32_t spg = static_cast<uint32_t>(p.nst / NG);  // stages of this group
      GroupRing gring;
      int buf = 0;
      for (int64_t t = t_begin + g; t < t_end; t += NG) {
        const int64_t w = GAIN ? qt.at(t, 0, p.W, 0) : 0;
        if (QUALITY) qual_window(p, qa, w, lane);
        if constexpr (GAIN)
          if (p.m_slots) enter(w);
        [[maybe_unused]] FrontierRows<S> fr;
        [[maybe_unused]] GainRows<S> gr;
        [[maybe_unused]] BaseRows<S> br;
        if constexpr (GAIN) gr.init(start_wide);
        else if constexpr (BASE) br.init();
        else fr.init();
        for (int k = 0; k < p.tiles_per_step; ++k) {
          const uint32_t st = gring.stage(g, NG), ph = gring.ph;
          gring.advance(spg);
          const bool have = mbar_wait_bounded(&full[st], ph, abort);
          unsigned char* tile = ring + size_t(st) * p.stage_bytes;
          // the tile's ranks; the last tile of a step starts early enough to be whole
          const int rank_fresh = k * p.tile_ranks;
          const int rank_tile0 = min(rank_fresh, R - p.tile_ranks);
          const int rank_end = rank_tile0 + p.tile_ranks;
          const int64_t first = t * RS + rank_tile0 * S;
          const int off = ALIGNED ? 0 : static_cast<int>(first & 15);
          if (!ALIGNED && have) patch_tail<kSwz>(tile, p.d, p.rows, first, p.tile_ranks * S, lane);
          if (have) {
            if constexpr (!GAIN) {
              for (int r0 = rank_fresh + ctid; r0 < rank_end; r0 += gthreads * U) {
                int64_t v[U][S];
  #pragma unroll
                for (int u = 0; u < U; ++u)
                  if (r0 + gthreads * u < rank_end) load_row<S, kSwz>(tile, off, r0 + gthreads * u - rank_tile0, v[u]);
  #pragma unroll
                for (int u = 0; u < U; ++u)
                  if (r0 + gthreads * u < rank_end) {
                    if constexpr (BASE) br.row(v[u], r0 + gthreads * u, dor, tor);
                    else fr.row(v[u], r0 + gthreads * u, dor, tor);
                  }
              }
            } else {
              // the medians of the same ranks: in the window's slot, or beside the tile
              unsigned char* mtile = tile + p.stage_bytes / 2;
              int64_t mfirst = w * RS + rank_tile0 * S;
              int mrank0 = rank_tile0;
              if (p.m_slots) {
                mtile = ms.base + size_t(place.slot(mwalk.at)) * p.m_bytes;
                mfirst = w * RS;
                mrank0 = 0;
              } else if constexpr (!ALIGNED) {
                patch_tail<kSwz>(mtile, p.m, p.m_rows, mfirst, p.tile_ranks * S, lane);
              }
              const int moff = ALIGNED ? 0 : static_cast<int>(mfirst & 15);
              if (m_have)
                for (int r = rank_fresh + ctid; r < rank_end; r += gthreads) {
                  const int q = r - rank_tile0, mq = r - mrank0;
                  const int64_t total = gr.row([&](int h) { return tile_pair<S, kSwz>(tile, off, q, h); },
                                               [&](int h) { return tile_pair<S, kSwz>(mtile, moff, mq, h); }, r, dor, tor);
                  if constexpr (QUALITY)
                    qual_row(p, qa, t, r, total, tile_stage<S, kSwz>(tile, off, q, p.other_stage), dor);
                }
            }
          }
          __syncwarp();
          if (lane == 0) mbar_arrive(&empty[st]);
        }
        // cross-rank reduction: warp redux, then one exchange through shared memory
        uint64_t* slot = red + (buf * kWarps + warp) * kRedPerWarp;
        uint64_t bslow = 0;
        [[maybe_unused]] bool narrow = false;
        if constexpr (BASE) bslow = warp_max_u64(br.slow);
        if constexpr (GAIN) {
          narrow = !__any_sync(kFull, gr.wide);
          start_wide = gr.met;
        }
  #pragma unroll
        for (int s = 0; s < S; ++s) {
          if constexpr (KIND == kFrontier) {
            const uint64_t km = warp_max_u64(fr.key(s));
            if (lane == s) slot[s] = km;
          } else if constexpr (BASE) {
            const uint64_t mx = warp_max_u64(static_cast<uint64_t>(br.mx[s]));
            const uint64_t sm = warp_sum_u64(br.sm[s]);
            if (lane == s) {
              slot[s] = mx;
              slot[S + s] = sm;
            }
          } else {
            uint64_t f, g;
            gr.warp_max(s, narrow, f, g);
            if (lane == s) {
              slot[s] = f;
              slot[S + s] = g;
            }
          }
        }
        if (BASE && lane == 0) slot[2 * S] = bslow;
        // the group's own barrier, its id an immediate operand
        switch (g) {
          case 0: named_barrier(1, gthreads); break;
          case 1: named_barrier(2, gthreads); break;
          case 2: named_barrier(3, gthreads); break;
          default: named_barrier(4, gthreads); break;
        }
        if (lw == 0) {
          uint64_t v0 = 0, v1 = 0, v2 = 0;
          if (lane < S) {
            for (int ww = warp; ww < warp + gw; ++ww) {
              const uint64_t* sl = red + (buf * kWarps + ww) * kRedPerWarp;
              v0 = sl[lane] > v0 ? sl[lane] : v0;
              if (GAIN) v1 = sl[S + lane] > v1 ? sl[S + lane] : v1;
              if (BASE) v1 += sl[S + lane];
            }
          }
          if (BASE) {
            for (int ww = warp; ww < warp + gw; ++ww) {
              const uint64_t k = red[(buf * kWarps + ww) * kRedPerWarp + 2 * S];
              v2 = k > v2 ? k : v2;
            }
          }
          if constexpr (KIND == kFrontier) finalize_frontier(p, S, t, v0, lane, acc);
          else if constexpr (BASE) finalize_base(p, S, t, v0, v1, v2, lane, bacc);
          else finalize_gain(p, S, t, w, v0, static_cast<int64_t>(v1), lane, acc);
        }
        buf ^= 1;
      }
    };
    if (p.groups == 4) consume(std::integral_constant<int, 4>{});
    else if (p.groups == 2) consume(std::integral_constant<int, 2>{});
    else consume(std::integral_constant<int, 1>{});
  }
  // no more steps: the producer may still wait for a slot that other warps need
  if constexpr (GAIN)
    if (p.m_slots && t_end > t_begin) {
      __syncwarp();
      mwalk.leave(static_cast<int>((t_end - 1) / p.W - w_base), p.m_slots, hand_back, landed);
    }

  const bool leader = p.regime == 0 || warp % (kWarps / p.groups) == 0;  // holds window accumulators
  if (BASE && leader) flush_base(p, S, bacc, lane);
  if (!BASE && p.X && leader) flush_window(p, S, acc, lane);
  if (QUALITY) qual_window(p, qa, -2, lane);
  const uint32_t bits = range_bits(__reduce_or_sync(kFull, dor), __reduce_or_sync(kFull, tor)) |
                        (*abort ? SF_ST_TIMEOUT : 0u);
  if (lane == 0) report(p.status, bits);
}

template <int KIND, bool ALIGNED>
cudaError_t dispatch_tiled(const CUtensorMap& map, const CUtensorMap& map_m, const Params& p, int grid,
                           cudaStream_t stream, bool pdl) {
  auto go = [&](auto s) -> cudaError_t {
    constexpr int S = decltype(s)::value;
    if constexpr (ALIGNED ? S % 2 == 0 : S != 16) {
      auto kern = stream_kernel<S, KIND, ALIGNED>;
      const size_t smem = tiled_smem(KIND, S, p.ring_bytes);
      const cudaError_t e =
          cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem));
      if (e != cudaSuccess) return e;
      return launch_ex(kern, grid, (consumer_warps(KIND, S) + kProducers) * 32, smem, stream, pdl, map, map_m, p);
    }
    return cudaErrorInvalidValue;
  };
  switch (p.S) {
#define SF_CASE(SV) \
  case SV: return go(std::integral_constant<int, SV>{});
    SF_CASE(1) SF_CASE(2) SF_CASE(3) SF_CASE(4) SF_CASE(5) SF_CASE(6) SF_CASE(7) SF_CASE(8)
    SF_CASE(9) SF_CASE(10) SF_CASE(11) SF_CASE(12) SF_CASE(13) SF_CASE(14) SF_CASE(15) SF_CASE(16)
#undef SF_CASE
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace
}  // namespace sf
