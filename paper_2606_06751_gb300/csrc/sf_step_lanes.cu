// sf_step_lanes.cu - the streaming passes with one lane per (step, stage), for
// small steps and for more than 16 stages.
//
// A warp takes 32 / S consecutive steps, lane j S + s stage s of the j-th, and
// walks their ranks together: per rank the lanes load their values (runs of S
// values per step, at any alignment), form the prefixes by a scan over their
// step's lanes, and each keeps its own stage's maxima.  Nothing is reduced
// across lanes until the step's end, so a step costs its ranks and one epilogue
// shared by all steps of the warp, where a warp per step pays S warp reductions
// for every step.  Loads are batched eight ranks deep
// (a second batch in flight cost four warps per SM and read slower).
//
// Values, medians and prefixes are taken in 32 bits; the tile (the warp's
// steps) is walked again in 64 bits when a value is 2^32 or more or the steps'
// per-stage maxima, which bound their prefixes, add up to that.  A warp that
// met such a tile walks the next one in 64 bits at once.
#include "sf_lane_select.cuh"
#include "sf_stream.cuh"

namespace sf {
namespace {

constexpr int kSlThreads = 128;
constexpr int kSlWarps = kSlThreads / 32;
constexpr int kSlBatch = 8;

// What a lane finds over the ranks of its step, for its stage.
struct LaneStep {
  int64_t F = 0;   // frontier
  int32_t lead = 0;
  int64_t G = 0;   // evidence: max_r (P_S - max(0, d - m))
  int64_t mx = 0;  // baselines: largest value, sum
  uint64_t sum = 0;
  uint64_t res = 0, ovl = 0, ws = 0;  // quality sums of the step, on its last stage's lane
  bool fits = true;                   // 32 bits hold the step
};

struct LanePlace {
  int j, s, last;  // step within the tile, stage, the lane of the step's last stage
  bool live;
};

template <int KIND, int LOGS, bool WIDE>
__device__ __forceinline__ LaneStep walk_ranks(const Params& p, const LanePlace& at, int64_t t, int64_t w, uint32_t& dor,
                                               uint32_t& tor) {
  constexpr bool GAIN = is_gain(KIND), QUALITY = KIND == kGainQuality, BASE = KIND == kBase;
  using V = std::conditional_t<WIDE, uint64_t, uint32_t>;
  const int S = static_cast<int>(p.S), R = static_cast<int>(p.R);
  const int64_t* col = p.d + t * p.R * p.S + at.s;
  [[maybe_unused]] const int64_t* mcol = GAIN ? p.m + w * p.R * p.S + at.s : nullptr;
  [[maybe_unused]] const bool walls = QUALITY && p.wall && at.live && at.s == S - 1;
  LaneStep o;
  V best = 0, g = 0;  // best: 1 + the largest prefix
  uint32_t lead = 0, high = 0, vmax = 0, dhi = 0;
  uint64_t vmax64 = 0;
  for (int r0 = 0; r0 < R; r0 += kSlBatch) {
    uint2 v[kSlBatch];
    [[maybe_unused]] uint2 mv[GAIN ? kSlBatch : 1], wv[QUALITY ? kSlBatch : 1];
#pragma unroll
    for (int i = 0; i < kSlBatch; ++i) {
      const int64_t r = min(r0 + i, R - 1);  // past the ranks: the last one again
      v[i] = load_words(col + r * S);
      if constexpr (GAIN) mv[i] = load_words(mcol + r * S);
      if constexpr (QUALITY) {
        wv[i] = make_uint2(0, 0);
        if (walls) wv[i] = load_words(p.wall + t * p.R + r);
      }
    }
#pragma unroll
    for (int i = 0; i < kSlBatch; ++i) {
      const int r = r0 + i;
      const V y = WIDE ? static_cast<V>((static_cast<uint64_t>(v[i].y) << 32) | v[i].x) : static_cast<V>(v[i].x);
      dhi |= v[i].y;
      if constexpr (WIDE) vmax64 = y > vmax64 ? y : vmax64;
      else vmax = max(vmax, static_cast<uint32_t>(y));
      V P = y;
#pragma unroll
      for (int q = 1; q < (1 << LOGS); q <<= 1) {
        const V up = __shfl_up_sync(kFull, P, q);
        if (at.s >= q) P += up;
      }
      const V P1 = P + 1;
      if (WIDE ? static_cast<int64_t>(P1) > static_cast<int64_t>(best) : P1 > best) {
        best = P1;
        lead = static_cast<uint32_t>(r);
      }
      if constexpr (GAIN) {
        const V total = __shfl_sync(kFull, P, at.last);
        const V m = WIDE ? static_cast<V>((static_cast<uint64_t>(mv[i].y) << 32) | mv[i].x) : static_cast<V>(mv[i].x);
        high |= mv[i].y;
        if constexpr (WIDE) {
          const int64_t cut = static_cast<int64_t>(y) > static_cast<int64_t>(m) ? static_cast<int64_t>(y - m) : 0;
          const int64_t alt = static_cast<int64_t>(total) - cut;
          g = alt > static_cast<int64_t>(g) ? static_cast<V>(alt) : g;
        } else {
          g = max(g, total - max(y, m) + m);
        }
      }
      if constexpr (BASE) o.sum += r < R ? static_cast<uint64_t>(y) : 0;
      if constexpr (QUALITY) {
        const V other = p.other_stage >= 0 ? __shfl_sync(kFull, y, at.last - (S - 1) + p.other_stage) : V(0);
        if (r < R) {
          const int64_t in = static_cast<int64_t>(P) - static_cast<int64_t>(other);  // the rank total but for `other`
          if (p.wall) {
            const int64_t wall = static_cast<int64_t>((static_cast<uint64_t>(wv[i].y) << 32) | wv[i].x);
            dor |= hi32(wall);
            const int64_t e = wall - in;
            if (e > 0) o.res += static_cast<uint64_t>(e);
            else o.ovl += static_cast<uint64_t>(-e);
            o.ws += static_cast<uint64_t>(wall);
          } else {
            o.res += static_cast<uint64_t>(other);
            o.ws += static_cast<uint64_t>(P);
          }
        }
      }
      if constexpr (WIDE)
        if (at.s == S - 1) tor |= static_cast<uint32_t>(static_cast<uint64_t>(P) >> 32);
    }
  }
  // would 32 bits hold every prefix?  The lanes' largest values bound them.
  uint64_t bound = WIDE ? (vmax64 >> 32 ? uint64_t(1) << 32 : vmax64) : vmax;
#pragma unroll
  for (int q = 1; q < (1 << LOGS); q <<= 1) {
    const uint64_t up = __shfl_up_sync(kFull, bound, q);
    if (at.s >= q) bound += up;
  }
  o.fits = (dhi | high) == 0 && ((bound + 1) >> 32) == 0;
  if constexpr (WIDE) dor |= dhi;
  o.F = static_cast<int64_t>(best) - 1;
  o.lead = static_cast<int32_t>(lead);
  o.G = static_cast<int64_t>(g);
  o.mx = static_cast<int64_t>(WIDE ? vmax64 : vmax);
  return o;
}

// Out of line: its registers do not weigh on the tiles that fit.
template <int KIND, int LOGS>
__device__ __noinline__ LaneStep walk_ranks_wide(const Params& p, const LanePlace& at, int64_t t, int64_t w,
                                                 uint32_t& dor, uint32_t& tor) {
  return walk_ranks<KIND, LOGS, true>(p, at, t, w, dor, tor);
}

// Largest key of a step's lanes, in all of them.
template <int LOGS>
__device__ __forceinline__ uint64_t step_max(uint64_t k, const LanePlace& at, int S) {
#pragma unroll
  for (int q = 1; q < (1 << LOGS); q <<= 1) {
    const uint64_t o = __shfl_down_sync(kFull, k, q);
    if (at.s + q < S && o > k) k = o;
  }
  return __shfl_sync(kFull, k, at.last - (S - 1));
}

template <int KIND, int LOGS>
__global__ void __launch_bounds__(kSlThreads, 5) step_lanes_kernel(const __grid_constant__ Params p) {
  constexpr bool GAIN = is_gain(KIND), QUALITY = KIND == kGainQuality, BASE = KIND == kBase;
  const int lane = threadIdx.x & 31;
  const int S = static_cast<int>(p.S);
  const int steps = 32 / S;  // per tile
  LanePlace at;
  at.j = lane / S;
  at.s = lane - at.j * S;
  at.last = min(at.j * S + S - 1, 31);
  const int64_t tiles = (p.T + steps - 1) / steps;
  const int64_t nw = int64_t(gridDim.x) * kSlWarps, id = int64_t(blockIdx.x) * kSlWarps + (threadIdx.x >> 5);
  const int64_t tile_end = tiles * (id + 1) / nw;
  uint32_t dor = 0, tor = 0;
  int64_t w = -1, w_end = 0;  // window of the lane's step: steps below w_end
  int64_t x = 0, y = 0, dsum = 0, slow = 0, r0 = 0;  // its sums so far (x: baselines' maxima)
  [[maybe_unused]] unsigned __int128 sum = 0, res = 0, ovl = 0, ws = 0;
  auto add = [&](int64_t* dst, int64_t v) {
    if (v) atomicAdd(reinterpret_cast<unsigned long long*>(dst), static_cast<unsigned long long>(v));
  };
  // The warp's window sums to global memory, those of one window over its steps first
  // (an atomic for every lane cost more than short runs: 12000 x 8 x 6 baselines 14.3 -> 8.2 us).
  auto flush = [&]() {
    const bool one = one_window(w);
    if (one) {
      x = sum_steps(x, S, lane);
      if constexpr (BASE) {
        sum = sum_steps(sum, S, lane);
        slow = sum_steps(slow, S, lane);
        r0 = sum_steps(r0, S, lane);
      } else {
        if constexpr (GAIN) y = sum_steps(y, S, lane);
        dsum = sum_steps(dsum, S, lane);
        if constexpr (QUALITY) {
          res = sum_steps(res, S, lane);
          ovl = sum_steps(ovl, S, lane);
          ws = sum_steps(ws, S, lane);
        }
      }
    }
    if (w >= 0 && (!one || lane < S)) {
      const int64_t i = w * S + at.s;
      if constexpr (BASE) {
        add(p.bM + i, x);
        if (sum) atomic_add_u128(p.bSUM + 2 * i, sum);
        add(p.bSLOW + i, slow);
        add(p.bRANK0 + i, r0);
      } else {
        add(p.X + i, x);
        if constexpr (GAIN) add(p.Y + i, y);
        if (at.s == S - 1) {
          add(p.D + w, dsum);
          if constexpr (QUALITY) {
            uint64_t* q = p.quality + w * 6;
            if (res) atomic_add_u128(q, res);
            if (ovl) atomic_add_u128(q + 2, ovl);
            if (ws) atomic_add_u128(q + 4, ws);
          }
        }
      }
    }
    x = y = dsum = slow = r0 = 0;
    if constexpr (BASE) sum = 0;
    if constexpr (QUALITY) res = ovl = ws = 0;
  };
  const bool windows = BASE || p.X;
  bool wide = false;  // walk the next tile in 64 bits at once
  griddep_wait();  // outputs cleared by the launch before this one (when it is its dependent)
  for (int64_t tile = tiles * id / nw; tile < tile_end; ++tile) {
    const int64_t t0 = tile * steps;
    at.live = at.j < steps && t0 + at.j < p.T;
    const int64_t t = at.live ? t0 + at.j : t0;
    const bool next = windows && at.live && (w < 0 || t >= w_end);
    if (__any_sync(kFull, next && w >= 0)) flush();
    if (next) {
      w = (p.t0 + t) / p.W - p.w_first;
      w_end = (w + p.w_first + 1) * p.W - p.t0;
    }
    const int64_t wm = GAIN ? (at.live ? w : t / p.W) : 0;
    LaneStep o;
    if (!wide) {
      o = walk_ranks<KIND, LOGS, false>(p, at, t, wm, dor, tor);
      wide = !__all_sync(kFull, o.fits);
      if (wide) o = walk_ranks_wide<KIND, LOGS>(p, at, t, wm, dor, tor);
    } else {
      o = walk_ranks_wide<KIND, LOGS>(p, at, t, wm, dor, tor);
      wide = !__all_sync(kFull, o.fits);
    }
    if constexpr (BASE) {
      // the slowest rank (largest total, lowest rank on ties) leads the last stage
      const int64_t rs = __shfl_sync(kFull, o.lead, at.last);
      if (at.live) {
        x += o.mx;
        sum += o.sum;
        slow += __ldg(p.d + (t * p.R + rs) * S + at.s);
        r0 += __ldg(p.d + t * p.R * S + at.s);
      }
      continue;
    }
    const int64_t before = __shfl_up_sync(kFull, o.F, 1);
    const int64_t a = o.F - (at.s ? before : 0);
    const int64_t FS = __shfl_sync(kFull, o.F, at.last);
    if (at.live) {
      if constexpr (!GAIN) {
        if (p.a) p.a[t * S + at.s] = a;
        if (p.lead) p.lead[t * S + at.s] = o.lead;
        if (p.mk && at.s == S - 1) p.mk[t] = o.F;
      }
      if (windows) {
        x += a;
        dsum += o.F;  // flushed by the last stage's lane
        if constexpr (GAIN) y += FS - o.G;
        if constexpr (QUALITY) {
          res += o.res;
          ovl += o.ovl;
          ws += o.ws;
        }
        const int64_t i = (w * S + at.s) * p.R + o.lead;
        if (p.E && a != 0) add(p.E + i, a);
        if (p.C) atomicAdd(p.C + i, 1);
      }
    }
    if (p.step_lead) {
      // leading stage (largest increment, lowest stage) and, for the evidence, the runner-up
      const uint64_t km = step_max<LOGS>((static_cast<uint64_t>(a) << 5) | static_cast<uint64_t>(31 - at.s), at, S);
      const int lead_stage = 31 - static_cast<int>(km & 31u);
      uint8_t code = static_cast<uint8_t>(lead_stage);
      if constexpr (GAIN) {
        const int64_t second = static_cast<int64_t>(step_max<LOGS>(at.s != lead_stage ? static_cast<uint64_t>(a) : 0, at, S));
        const bool conf = FS > 0 && static_cast<__int128>(static_cast<int64_t>(km >> 5) - second) * p.eta_den >=
                                        static_cast<__int128>(p.eta_num) * FS;
        if (conf) code |= SF_STEP_CONFIDENT;
      }
      if (at.live && at.s == 0) p.step_lead[t] = code;
    }
  }
  if (windows) flush();
  const uint32_t bits = range_bits(__reduce_or_sync(kFull, dor), __reduce_or_sync(kFull, tor));
  if (lane == 0) report(p.status, bits);
}

template <int KIND, int LOGS>
cudaError_t launch_logs(const Params& p, cudaStream_t stream, bool pdl) {
  auto kern = step_lanes_kernel<KIND, LOGS>;
  int per_sm = 1;
  const cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kSlThreads, 0);
  if (e != cudaSuccess) return e;
  const int64_t tiles = (p.T + 32 / p.S - 1) / (32 / p.S);
  const int64_t grid = std::min<int64_t>((tiles + kSlWarps - 1) / kSlWarps, int64_t(sm_count()) * std::max(per_sm, 1));
  return launch_ex(kern, dim3(static_cast<unsigned>(grid)), kSlThreads, 0, stream, pdl, p);
}

template <int KIND>
cudaError_t launch_kind(const Params& p, cudaStream_t stream, bool pdl) {
  if (p.S <= 1) return launch_logs<KIND, 0>(p, stream, pdl);
  if (p.S <= 2) return launch_logs<KIND, 1>(p, stream, pdl);
  if (p.S <= 4) return launch_logs<KIND, 2>(p, stream, pdl);
  if (p.S <= 8) return launch_logs<KIND, 3>(p, stream, pdl);
  if (p.S <= 16) return launch_logs<KIND, 4>(p, stream, pdl);
  if constexpr (is_gain(KIND))
    return launch_logs<KIND, 5>(p, stream, pdl);
  else
    return cudaErrorInvalidValue;  // use_step_lanes: only evidence takes more than 16 stages here
}

}  // namespace

cudaError_t launch_step_lanes(int kind, const Params& p, cudaStream_t stream, bool pdl) {
  switch (kind) {
    case kFrontier: return launch_kind<kFrontier>(p, stream, pdl);
    case kGain: return launch_kind<kGain>(p, stream, pdl);
    case kGainQuality: return launch_kind<kGainQuality>(p, stream, pdl);
    default: return launch_kind<kBase>(p, stream, pdl);
  }
}

}  // namespace sf
