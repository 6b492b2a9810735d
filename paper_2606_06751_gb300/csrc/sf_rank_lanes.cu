// sf_rank_lanes.cu - cross-rank order statistics of steps with few ranks: one
// lane per (step, stage) column (see sf_rank_chip.cu).
//
// A warp takes 32 / S consecutive steps, lane j S + s stage s of the j-th.  Per
// rank the lanes load their values (runs of S values per step), form the
// prefixes by a scan over their step's lanes, and keep the low words as keys in
// registers; minimum, the two largest and the median are then each lane's own
// affair.  Prefixes fit 32 bits when every value does and the step's per-stage
// maxima add up to less than 2^32 ns; another step is taken again by the whole
// warp on 64-bit values, column by column.
#include "sf_lane_select.cuh"
#include "sf_rank_chip.cuh"

namespace sf {
namespace {

constexpr int kLaneThreads = 128;
constexpr int kLaneWarps = kLaneThreads / 32;

struct WideScratch {  // of one warp
  uint32_t hist[256];
  int64_t col[kRankLaneMax];
};

// A step on 64-bit values by the whole warp: lane s gets column s's statistics.
__device__ __noinline__ void wide_step(const int64_t* dt, int R, int S, bool of_prefix, int lane, WideScratch& sc,
                                       int64_t& med, int64_t& top, int64_t& second, uint32_t& tor) {
  constexpr int kPer = kRankLaneMax / 32;
  int64_t run[kPer];
#pragma unroll
  for (int i = 0; i < kPer; ++i) run[i] = 0;
#pragma unroll 1
  for (int s = 0; s < S; ++s) {
#pragma unroll
    for (int i = 0; i < kPer; ++i) {
      const int r = lane + 32 * i;
      if (r >= R) break;
      const int64_t v = __ldg(dt + int64_t(r) * S + s);
      run[i] = of_prefix ? run[i] + v : v;
      sc.col[r] = run[i];
    }
    __syncwarp();
    int64_t a, b, c;
    column_64(sc.col, R, sc.hist, lane, a, b, c);
    if (lane == s) {
      med = a;
      top = b;
      second = c;
    }
    __syncwarp();
  }
  if (of_prefix)
#pragma unroll
    for (int i = 0; i < kPer; ++i) tor |= hi32(run[i]);
}

// The per-step state beside the keys costs a CTA more than the median's lanes.
constexpr int rank_lane_ctas(int nmax) { return nmax <= 32 ? 4 : nmax <= 64 ? 3 : 2; }

// LOGS: scan rounds that form the prefixes, ceil(log2 S); 0 for the durations.
template <int NMAX, int LOGS>
__global__ void __launch_bounds__(kLaneThreads, rank_lane_ctas(NMAX)) rank_lanes_kernel(const ChipParams p) {
  __shared__ WideScratch scratch[kLaneWarps];
  constexpr int kBatch = lane_batch(NMAX);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int S = p.S, R = p.R;
  const int steps = 32 / S;  // per tile
  const int j = lane / S, s = lane - j * S;
  const int64_t tiles = (p.T + steps - 1) / steps;
  const int64_t nw = int64_t(gridDim.x) * kLaneWarps, id = int64_t(blockIdx.x) * kLaneWarps + warp;
  const int64_t tile_end = tiles * (id + 1) / nw;
  const uint32_t n = static_cast<uint32_t>(R), kth = (n - 1) / 2;
  const bool windows = p.Lw || p.Gw || p.spread;
  uint32_t dor = 0, tor = 0;
  int64_t w = -1, w_end = 0;   // window of the lane's step: steps below w_end
  int64_t accL = 0, accG = 0;  // its sums so far
  auto flush = [&]() {
    if (w < 0) return;
    if (p.Lw) add_window(p.Lw, w * S + s, accL);
    if (p.Gw) add_window(p.Gw, w * S + s, accG);
    if (p.spread) add_window(p.spread, w * S + s, accL);
  };
  for (int64_t tile = tiles * id / nw; tile < tile_end; ++tile) {
    const int64_t t0 = tile * steps, t = t0 + j;
    const bool live = j < steps && t < p.T;
    const int64_t* col = p.d + (live ? t : t0) * R * S + s;
    if (lane == 0 && tile + 1 < tile_end)
      prefetch_step(p.d + (t0 + steps) * R * S, (min(t0 + 2 * steps, p.T) - t0 - steps) * R * S);
    uint32_t x[NMAX];
    uint32_t hor = 0, vmax = 0;
#pragma unroll
    for (int b = 0; b < NMAX; b += kBatch) {
      uint2 v[kBatch];
#pragma unroll
      for (int i = 0; i < kBatch; ++i) v[i] = load_words(col + min(b + i, R - 1) * S);  // past the ranks: the last one
#pragma unroll
      for (int i = 0; i < kBatch; ++i) {
        hor |= v[i].y;
        uint32_t y = v[i].x;
        vmax = max(vmax, y);
#pragma unroll
        for (int o = 1; o < (1 << LOGS); o <<= 1) {
          const uint32_t up = __shfl_up_sync(kFull, y, o);
          if (s >= o) y += up;
        }
        x[b + i] = b + i < R ? y : 0xffffffffu;  // sorts last
      }
    }
    dor |= hor;
    // steps whose keys do not hold: a value, or the bound on the totals, past 32 bits
    uint64_t bound = vmax;
#pragma unroll
    for (int o = 1; o < (1 << LOGS); o <<= 1) {
      const uint64_t up = __shfl_up_sync(kFull, bound, o);
      if (s >= o) bound += up;
    }
    const uint32_t wide = __ballot_sync(kFull, live && (hor != 0 || (bound >> 32) != 0));
    uint32_t lo = 0xffffffffu, k1 = 0, k2 = 0;
#pragma unroll
    for (int i = 0; i < NMAX; ++i) {
      lo = min(lo, x[i]);
      top2_add(k1, k2, i < R ? x[i] : 0u);
    }
    if (R < 2) k2 = k1;
    int64_t med = lane_select<NMAX>(x, n, kth, lo, k1), top = k1, second = k2;
    for (int q = 0; wide != 0 && q < steps; ++q) {
      if (!(wide & (((S == 32 ? 0u : 1u << S) - 1u) << (q * S)))) continue;
      int64_t a, b, c;
      wide_step(p.d + (t0 + q) * R * S, R, S, p.of_prefix, lane, scratch[warp], a, b, c, tor);
      const int64_t ma = __shfl_sync(kFull, a, s), mb = __shfl_sync(kFull, b, s), mc = __shfl_sync(kFull, c, s);
      if (j == q) {
        med = ma;
        top = mb;
        second = mc;
      }
    }
    const int64_t lag = top - med, gap = top - second;
    const int64_t before = __shfl_up_sync(kFull, lag, 1);
    if (live) {
      if (p.L) p.L[t * S + s] = lag;
      if (p.dL) p.dL[t * S + s] = lag - (s ? before : 0);
      if (p.G) p.G[t * S + s] = gap;
      if (windows) {
        if (w < 0 || t >= w_end) {
          flush();
          w = (p.t0 + t) / p.W - p.w_first;
          w_end = (w + p.w_first + 1) * p.W - p.t0;
          accL = accG = 0;
        }
        accL += lag;
        accG += gap;
      }
    }
  }
  if (windows) flush();
  const uint32_t bits = range_bits(__reduce_or_sync(kFull, dor), p.of_prefix ? __reduce_or_sync(kFull, tor) : 0u);
  if (lane == 0) report(p.status, bits);
}

template <int LOGS>
cudaError_t launch_lanes(const ChipParams& p, cudaStream_t stream) {
  auto go = [&](auto kern) { return launch_chip(kern, p, kLaneThreads, 0, int64_t(kLaneWarps) * (32 / p.S), stream); };
  if (p.R <= 16) return go(rank_lanes_kernel<16, LOGS>);
  if (p.R <= 32) return go(rank_lanes_kernel<32, LOGS>);
  if (p.R <= 64) return go(rank_lanes_kernel<64, LOGS>);
  if (p.R <= 104) return go(rank_lanes_kernel<104, LOGS>);
  return go(rank_lanes_kernel<128, LOGS>);
}

}  // namespace

cudaError_t launch_rank_lanes(const ChipParams& p, cudaStream_t stream) {
  if (!p.of_prefix || p.S == 1) return launch_lanes<0>(p, stream);
  if (p.S <= 2) return launch_lanes<1>(p, stream);
  if (p.S <= 4) return launch_lanes<2>(p, stream);
  if (p.S <= 8) return launch_lanes<3>(p, stream);
  if (p.S <= 16) return launch_lanes<4>(p, stream);
  return launch_lanes<5>(p, stream);
}

}  // namespace sf
