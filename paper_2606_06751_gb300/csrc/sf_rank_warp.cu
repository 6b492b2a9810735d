// sf_rank_warp.cu - cross-rank order statistics of steps of 65 to 128 ranks and
// up to 8 stages: one warp per step, the step's keys in registers (see
// sf_rank_chip.cu).
#include <type_traits>

#include "sf_rank_chip.cuh"

namespace sf {
namespace {

constexpr int kWarpThreads = 256;

struct WarpScratch {  // of one warp, for steps that do not fit 32 bits
  uint32_t hist[256];
  int64_t ref[kChipMaxS];
  int64_t col[256];
};

struct StepStats {  // lane s: of column s
  int64_t med, top, second;
};

// One step by one warp.  REL = false: the values' low words are the keys;
// returns false, without a result, when they do not fit 32 bits.  REL = true:
// the step again, relative to rank 0's values or in 64 bits.
template <int S, int NPL, bool VEC, bool REL>
__device__ __forceinline__ bool warp_step(const int64_t* dt, int R, bool of_prefix, int lane,
                                          WarpScratch& sc, StepStats& o, uint32_t& dor, uint32_t& tor) {
  const uint32_t kth = static_cast<uint32_t>((R - 1) / 2);
  uint32_t k[S][NPL];
  uint32_t wide = 0;
#pragma unroll
  for (int i = 0; i < NPL; ++i) {
    const int r = lane + 32 * i;
    const bool live = r < R;
    int64_t v[S];
    const int64_t* row = dt + int64_t(live ? r : 0) * S;
    if constexpr (VEC) {
#pragma unroll
      for (int s = 0; s < S; s += 2) {
        const longlong2 x = __ldg(reinterpret_cast<const longlong2*>(row + s));
        v[s] = x.x;
        v[s + 1] = x.y;
      }
    } else {
#pragma unroll
      for (int s = 0; s < S; ++s) {
        v[s] = __ldg(row + s);
      }
    }
    uint64_t P = 0;
    uint32_t vh = 0;
#pragma unroll
    for (int s = 0; s < S; ++s) {
      vh |= hi32(v[s]);
      P += static_cast<uint64_t>(v[s]);
      const uint32_t x = of_prefix ? static_cast<uint32_t>(P) : static_cast<uint32_t>(v[s]);
      k[s][i] = live ? x : 0xffffffffu;  // a missing rank sorts last
    }
    dor |= vh;
    const uint32_t th = static_cast<uint32_t>(P >> 32);
    tor |= th;
    wide |= vh | (of_prefix ? th : 0u);
  }
  // lane s: what column s's keys are relative to
  [[maybe_unused]] int64_t ref = 0;
  if constexpr (!REL) {
    if (__any_sync(kFull, wide != 0)) return false;
  } else {
    ref = lane < S ? step_value(dt, S, of_prefix, 0, lane) : 0;
    if (lane < S) sc.ref[lane] = ref;
    __syncwarp();
    const bool far = __any_sync(kFull, far_from_first(dt, R, S, of_prefix, sc.ref, lane, 32));
    __syncwarp();
    if (far) {
      int64_t run[NPL];
#pragma unroll
      for (int i = 0; i < NPL; ++i) run[i] = 0;
#pragma unroll 1
      for (int s = 0; s < S; ++s) {
#pragma unroll
        for (int i = 0; i < NPL; ++i) {
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
          o.med = a;
          o.top = b;
          o.second = c;
        }
      }
      return true;
    }
    const uint32_t bias = static_cast<uint32_t>(ref) - kSign32;
#pragma unroll
    for (int s = 0; s < S; ++s) {
      const uint32_t b = __shfl_sync(kFull, bias, s);
#pragma unroll
      for (int i = 0; i < NPL; ++i)
        if (lane + 32 * i < R) k[s][i] -= b;
    }
  }
  uint32_t lo = 0, hi = 0, k2 = 0;
#pragma unroll
  for (int s = 0; s < S; ++s) {
    uint32_t mn = k[s][0], a1 = lane < R ? k[s][0] : 0u, a2 = 0u;
#pragma unroll
    for (int i = 1; i < NPL; ++i) {
      mn = min(mn, k[s][i]);
      top2_add(a1, a2, lane + 32 * i < R ? k[s][i] : 0u);
    }
    mn = __reduce_min_sync(kFull, mn);
    warp_top2(a1, a2);
    if (lane == s) {
      lo = mn;
      hi = a1;
      k2 = a2;
    }
  }
  const uint32_t k1 = hi;
  // the median is in [lo, hi]; below keys lie under lo, upto at or under hi
  uint32_t below = 0, upto = static_cast<uint32_t>(R);
  for (uint32_t round = 0;; ++round) {
    const bool open = lane < S && lo < hi && below != kth && upto != kth + 1;
    const uint32_t open_mask = __ballot_sync(kFull, open);
    if (open_mask == 0) break;
    // every second round probes where the median would lie if the keys
    // were spread evenly over the bracket
    const uint32_t span = hi - lo;
    uint32_t mid = lo + (span >> 1);
    if (round & 1u) {
      const float at = __fdividef(static_cast<float>(kth - below) + 0.5f, static_cast<float>(upto - below));
      mid = lo + min(static_cast<uint32_t>(at * static_cast<float>(span)), span - 1u);
    }
    uint32_t cnt = 0;
#pragma unroll
    for (int s = 0; s < S; ++s) {
      if (!((open_mask >> s) & 1u)) continue;
      const uint32_t m = __shfl_sync(kFull, mid, s);
      uint32_t c = 0;
#pragma unroll
      for (int i = 0; i < NPL; ++i) c += k[s][i] <= m ? 1u : 0u;
      c = __reduce_add_sync(kFull, c);
      if (lane == s) cnt = c;
    }
    if (open) {
      if (cnt > kth) {
        hi = mid;
        upto = cnt;
      } else {
        lo = mid + 1;
        below = cnt;
      }
    }
  }
  uint32_t ans = lo;
  const uint32_t low_mask = __ballot_sync(kFull, lane < S && lo < hi && below == kth);
  const uint32_t high_mask = __ballot_sync(kFull, lane < S && lo < hi && below != kth);
#pragma unroll
  for (int s = 0; s < S; ++s) {
    if ((low_mask >> s) & 1u) {  // the smallest key from lo on
      const uint32_t m = __shfl_sync(kFull, lo, s);
      uint32_t x = 0xffffffffu;
#pragma unroll
      for (int i = 0; i < NPL; ++i) x = min(x, k[s][i] >= m ? k[s][i] : 0xffffffffu);
      x = __reduce_min_sync(kFull, x);
      if (lane == s) ans = x;
    } else if ((high_mask >> s) & 1u) {  // the largest key up to hi
      const uint32_t m = __shfl_sync(kFull, hi, s);
      uint32_t x = 0;
#pragma unroll
      for (int i = 0; i < NPL; ++i) x = max(x, k[s][i] <= m ? k[s][i] : 0u);
      x = __reduce_max_sync(kFull, x);
      if (lane == s) ans = x;
    }
  }
  if (R < 2) k2 = k1;
  auto value = [&](uint32_t key) {
    return REL ? ref + static_cast<int64_t>(static_cast<int32_t>(key ^ kSign32)) : static_cast<int64_t>(key);
  };
  o.med = value(ans);
  o.top = value(k1);
  o.second = value(k2);
  return true;
}

// Out of line: its registers and code do not weigh on the steps that fit.
template <int S, int NPL, bool VEC>
__device__ __noinline__ void warp_step_rel(const int64_t* dt, int R, bool of_prefix, int lane, WarpScratch& sc,
                                           StepStats& o) {
  uint32_t dor = 0, tor = 0;
  warp_step<S, NPL, VEC, true>(dt, R, of_prefix, lane, sc, o, dor, tor);
}

// NPL >= ceil(R / 32): the ranks per lane; VEC: S even, rows read 16 bytes at a time.
template <int S, int NPL, bool VEC>
__global__ void __launch_bounds__(kWarpThreads, 3) rank_warp_kernel(const ChipParams p) {
  __shared__ WarpScratch scratch[kWarpThreads / 32];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int R = p.R;
  const int64_t nw = int64_t(gridDim.x) * (kWarpThreads / 32), id = int64_t(blockIdx.x) * (kWarpThreads / 32) + warp;
  const int64_t t_begin = p.T * id / nw, t_end = p.T * (id + 1) / nw;
  uint32_t dor = 0, tor = 0;
  int64_t w = -1, w_end = 0;      // window of the step: steps below w_end
  int64_t accL = 0, accG = 0;     // its sums so far, lane s for stage s
  auto flush = [&]() {
    if (w < 0 || lane >= S) return;
    if (p.of_prefix) {
      if (p.Lw) add_window(p.Lw, w * S + lane, accL);
      if (p.Gw) add_window(p.Gw, w * S + lane, accG);
    } else {
      add_window(p.spread, w * S + lane, accL);
    }
  };
  const bool windows = p.Lw || p.Gw || p.spread;
  for (int64_t t = t_begin; t < t_end; ++t) {
    const int64_t* dt = p.d + t * R * S;
    if (lane == 0 && t + 1 < t_end) prefetch_step(dt + R * S, R * S);
    StepStats o;
    if (!warp_step<S, NPL, VEC, false>(dt, R, p.of_prefix, lane, scratch[warp], o, dor, tor))
      warp_step_rel<S, NPL, VEC>(dt, R, p.of_prefix, lane, scratch[warp], o);
    const int64_t lag = o.top - o.med, gap = o.top - o.second;
    const int64_t before = __shfl_up_sync(kFull, lag, 1);
    if (lane < S) {
      if (p.L) p.L[t * S + lane] = lag;
      if (p.dL) p.dL[t * S + lane] = lag - (lane ? before : 0);
      if (p.G) p.G[t * S + lane] = gap;
    }
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
  if (windows) flush();
  const uint32_t bits = range_bits(__reduce_or_sync(kFull, dor), p.of_prefix ? __reduce_or_sync(kFull, tor) : 0u);
  if (lane == 0) report(p.status, bits);
}

}  // namespace

cudaError_t launch_rank_warp(const ChipParams& p, cudaStream_t stream) {
  auto go = [&](auto s) {
    constexpr int S = decltype(s)::value;
    return launch_chip(rank_warp_kernel<S, kRankLaneMax / 32, S % 2 == 0>, p, kWarpThreads, 0, kWarpThreads / 32, stream);
  };
  switch (p.S) {
#define SF_CASE(SV) \
  case SV: return go(std::integral_constant<int, SV>{});
    SF_CASE(1) SF_CASE(2) SF_CASE(3) SF_CASE(4) SF_CASE(5) SF_CASE(6) SF_CASE(7) SF_CASE(8)
#undef SF_CASE
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace sf
