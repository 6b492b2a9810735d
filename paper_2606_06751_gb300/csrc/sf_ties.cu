// sf_ties.cu - size of the lead rank's tie set per step and stage (Sec. 4:
// among the localization evidence the labeler reports the latest-rank tie
// set): ties[t,s] = #{r : P[t,r,s] = F[t,s]}, the ranks whose prefix reaches
// the frontier.  1 means the lead rank is the unique one; more means a tie
// that the frontier pass resolved to the lowest rank.
//
// One more pass over d: per step, the frontier F[t,s] is rebuilt from the
// increments a[t,.] of the frontier pass (their prefix over s), every thread
// counts, per stage, its rank rows whose prefix equals it, and the counts are
// summed.  Three splits of the work, chosen by launch_frontier_ties:
//   ties_warp_kernel - a warp per step, no CTA barrier, for small steps that are
//     many enough.  Three barriers a step bound them (100000 x 128 x 8: 344 us with a
//     CTA per step, 136 us, 90 % of the measured copy rate, with a warp);
//   ties_kernel      - a CTA per step, the CTA walking a range of steps; with
//     fewer steps than the chip holds CTAs, a thread-block cluster per step,
//     its CTAs' counts summed through distributed shared memory (one step of
//     8192 x 8: 19.8 us in one CTA, 8.3 us in a cluster of eight).
// The per-stage state is sized by a bound SMAX >= S with every stage loop
// unrolled to SMAX behind an `s < S` test, so it stays in registers.
#include <algorithm>
#include <type_traits>

#include <cooperative_groups.h>

#include "sf_device.cuh"
#include "sf_launch.h"

namespace sf {

namespace {

constexpr int kTieThreads = 256;
constexpr int kTieWarps = kTieThreads / 32;
constexpr int kTieCluster = 8;

// Resident ties_kernel CTAs per SM.
__host__ __device__ constexpr int tie_ctas(int smax, bool staged) { return smax <= 8 ? 4 : smax == 32 || staged ? 2 : 3; }

// Whether a step takes a warp.  A lane walks R / 32 rows alone, so the longer that is
// the more warps per SM it takes to beat a CTA per step (us, CTA / warp: 600 x 100 x 3
// 4.2 / 6.2, 800 x 100 x 3 6.2 / 6.2, 2500 x 100 x 3 8.2 / 6.2; 1200 x 330 x 6 8.3 / 10.3, 2500 x 330 x 6
// 12.4 / 10.3; 1200 x 330 x 14 14.4 / 12.3; 2500 x 500 x 20 73.9 / 85.8).
bool use_warps(int64_t T, int64_t R, int64_t S, int64_t sms) {
  if (R <= 32) return true;
  if (R <= 128) return T >= sms * (R > 64 && S <= 8 ? 8 : 4);
  if (S > 16) return R <= 340 && T >= sms * 5;
  return R <= 512 && T >= sms * (S <= 8 ? 12 : 5);
}

__device__ __forceinline__ uint32_t hi32(int64_t v) {
  return static_cast<uint32_t>(static_cast<uint64_t>(v) >> 32);
}

// Lane s < S: F[t,s], the inclusive prefix of the increments over s.
__device__ __forceinline__ int64_t lane_frontier(const int64_t* a, int64_t t, int S, int lane) {
  int64_t x = lane < S ? __ldg(a + t * S + lane) : 0;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int64_t up = __shfl_up_sync(kFull, x, o);
    if (lane >= o) x += up;
  }
  return x;
}

// Counts the rows r0, r0 + stride, ... < r1 of a step whose prefix equals F.
// VEC: S even, rows start 16-byte aligned and are read with 16-byte loads.  With
// 9 to 16 stages a row's loads are all issued before its first use (50000 x 1024 x
// 10: 1100 -> 846 us); shorter rows gain nothing by it, longer ones cost too many
// registers (1000 x 24: 141 against 189 us).
template <int SMAX, bool VEC, bool STAGED = SMAX == 16>
__device__ __forceinline__ void count_rows(const int64_t* dt, int S, int r0, int r1, int stride,
                                           const int64_t (&F)[SMAX], uint32_t (&cnt)[SMAX], uint32_t& dor,
                                           uint32_t& tor) {
  constexpr int kStage = STAGED ? SMAX : VEC ? 2 : 1;  // stages loaded together
  for (int r = r0; r < r1; r += stride) {
    const int64_t* row = dt + int64_t(r) * S;
    int64_t P = 0;
#pragma unroll
    for (int s0 = 0; s0 < SMAX; s0 += kStage) {
      if (s0 >= S) break;
      int64_t v[kStage];
#pragma unroll
      for (int i = 0; i < kStage; i += VEC ? 2 : 1) {
        if (s0 + i >= S) break;
        if constexpr (VEC) {
          const longlong2 x = __ldg(reinterpret_cast<const longlong2*>(row + s0 + i));
          v[i] = x.x;
          v[i + 1] = x.y;
        } else {
          v[i] = __ldg(row + s0 + i);
        }
      }
#pragma unroll
      for (int i = 0; i < kStage; ++i) {
        if (s0 + i >= S) break;
        dor |= hi32(v[i]);
        P += v[i];
        cnt[s0 + i] += P == F[s0 + i] ? 1u : 0u;
      }
    }
    tor |= hi32(P);
  }
}

template <int SMAX, bool VEC>
__global__ void __launch_bounds__(kTieThreads)
    ties_warp_kernel(const int64_t* __restrict__ d, int64_t T, int R, int S, const int64_t* __restrict__ a,
                     int32_t* __restrict__ ties, uint32_t* status) {
  const int lane = threadIdx.x & 31;
  const int64_t nw = int64_t(gridDim.x) * kTieWarps, id = int64_t(blockIdx.x) * kTieWarps + (threadIdx.x >> 5);
  uint32_t dor = 0, tor = 0;
  for (int64_t t = id; t < T; t += nw) {
    const int64_t x = lane_frontier(a, t, S, lane);
    int64_t F[SMAX];
    uint32_t cnt[SMAX];
#pragma unroll
    for (int s = 0; s < SMAX; ++s) {
      if (s >= S) break;
      F[s] = __shfl_sync(kFull, x, s);
      cnt[s] = 0;
    }
    count_rows<SMAX, VEC>(d + t * R * S, S, lane, R, 32, F, cnt, dor, tor);
    uint32_t mine = 0;
#pragma unroll
    for (int s = 0; s < SMAX; ++s) {
      if (s >= S) break;
      const uint32_t c = __reduce_add_sync(kFull, cnt[s]);
      if (lane == s) mine = c;
    }
    if (lane < S) ties[t * S + lane] = static_cast<int32_t>(mine);
  }
  const uint32_t bits = range_bits(__reduce_or_sync(kFull, dor), __reduce_or_sync(kFull, tor));
  if (lane == 0) report(status, bits);
}

// A CTA per step or, with SPLIT, a cluster of CTAs, each counting an equal share of
// the ranks.
template <int SMAX, bool VEC, bool SPLIT, bool STAGED = SMAX == 16>
__global__ void __launch_bounds__(kTieThreads, tie_ctas(SMAX, STAGED))
    ties_kernel(const int64_t* __restrict__ d, int64_t T, int R, int S, const int64_t* __restrict__ a,
                int32_t* __restrict__ ties, uint32_t* status) {
  namespace cg = cooperative_groups;
  __shared__ int64_t sF[32];
  __shared__ uint32_t wcnt[kTieWarps][32];
  __shared__ uint32_t sum[32];
  const int csize = SPLIT ? static_cast<int>(cg::this_cluster().num_blocks()) : 1;
  const int part = SPLIT ? static_cast<int>(cg::this_cluster().block_rank()) : 0;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t NB = gridDim.x / csize, b = blockIdx.x / csize;
  const int64_t t_begin = T * b / NB, t_end = T * (b + 1) / NB;
  const int r0 = static_cast<int>(int64_t(R) * part / csize), r1 = static_cast<int>(int64_t(R) * (part + 1) / csize);
  uint32_t dor = 0, tor = 0;
  for (int64_t t = t_begin; t < t_end; ++t) {
    if (warp == 0) {
      const int64_t x = lane_frontier(a, t, S, lane);
      if (lane < S) sF[lane] = x;
    }
    __syncthreads();
    int64_t F[SMAX];
    uint32_t cnt[SMAX];
#pragma unroll
    for (int s = 0; s < SMAX; ++s) {
      if (s >= S) break;
      F[s] = sF[s];
      cnt[s] = 0;
    }
    count_rows<SMAX, VEC, STAGED>(d + t * R * S, S, r0 + static_cast<int>(threadIdx.x), r1, kTieThreads, F, cnt, dor, tor);
#pragma unroll
    for (int s = 0; s < SMAX; ++s) {
      if (s >= S) break;
      const uint32_t c = __reduce_add_sync(kFull, cnt[s]);
      if (lane == 0) wcnt[warp][s] = c;
    }
    __syncthreads();
    uint32_t c = 0;
    if (warp == 0 && lane < S) {
#pragma unroll
      for (int w = 0; w < kTieWarps; ++w) c += wcnt[w][lane];
      sum[lane] = c;
    }
    if constexpr (SPLIT) {
      cg::cluster_group cluster = cg::this_cluster();
      cluster.sync();  // every CTA's counts are written
      if (part == 0 && warp == 0 && lane < S)
        for (int q = 1; q < csize; ++q) c += *cluster.map_shared_rank(&sum[lane], static_cast<unsigned>(q));
      cluster.sync();  // ... and read, before a CTA leaves or writes its next step's
    }
    if (part == 0 && warp == 0 && lane < S) ties[t * S + lane] = static_cast<int32_t>(c);
    __syncthreads();  // sF and wcnt are rewritten for the next step
  }
  const uint32_t bits = range_bits(__reduce_or_sync(kFull, dor), __reduce_or_sync(kFull, tor));
  if (lane == 0) report(status, bits);
}

}  // namespace

cudaError_t launch_frontier_ties(const int64_t* d, int64_t T, int64_t R, int64_t S, const int64_t* a,
                                 int32_t* ties, uint32_t* status, cudaStream_t stream) {
  const int s = static_cast<int>(S), r = static_cast<int>(R);
  count_launch();
  auto go = [&](auto smax, auto vec) {
    constexpr int SM = decltype(smax)::value;
    constexpr bool V = decltype(vec)::value;
    const int64_t sms = sm_count();
    if (use_warps(T, R, S, sms)) {
      const int grid = static_cast<int>(std::min<int64_t>(sms * 8, (T + kTieWarps - 1) / kTieWarps));
      ties_warp_kernel<SM, V><<<grid, kTieThreads, 0, stream>>>(d, T, r, s, a, ties, status);
      return cudaGetLastError();
    }
    // few large steps: CTAs of a cluster share one, each with at least two rows a thread
    // (100 x 1064 x 2 4.2 us in one CTA, 6.2 in two; 100 x 4217 x 6 12.3 / 8.3).  Clusters of
    // four and more need room to be placed (152 x 8192 x 8 in four, filling every slot, 21.6
    // us, in two 18.4; 76 x 15000 x 32 in four 137, in two 117)
    const int64_t ctas = sms * (SM <= 8 ? 4 : 2);
    unsigned csize = 1;
    if (R * S * 8 >= 72 * 1024)
      while (csize < kTieCluster && T * csize * 2 <= (csize > 1 ? ctas * 7 / 8 : ctas) &&
             R >= int64_t(csize) * 4 * kTieThreads)
        csize *= 2;
    if (csize == 1) {
      // staged rows hold two CTAs per SM: a few more steps than those run in one round
      // of three without (330 x 1064 x 14 14.3 us staged, 12.3 not; 600 x 1064 x 14 14.4, 20.5)
      if constexpr (SM == 16)
        if (T > ctas && T <= sms * tie_ctas(SM, false)) {
          ties_kernel<SM, V, false, false><<<static_cast<unsigned>(T), kTieThreads, 0, stream>>>(d, T, r, s, a, ties, status);
          return cudaGetLastError();
        }
      const int grid = static_cast<int>(std::min<int64_t>(SM == 32 ? sms * 4 : ctas, T));
      ties_kernel<SM, V, false><<<grid, kTieThreads, 0, stream>>>(d, T, r, s, a, ties, status);
      return cudaGetLastError();
    }
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = csize;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(static_cast<unsigned>(std::min<int64_t>(ctas / csize, T) * csize));
    cfg.blockDim = dim3(kTieThreads);
    cfg.stream = stream;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, ties_kernel<SM, V, true>, d, T, r, s, a, ties, status);
  };
  auto pick = [&](auto smax) {
    return S % 2 == 0 ? go(smax, std::true_type{}) : go(smax, std::false_type{});
  };
  if (S <= 4) return pick(std::integral_constant<int, 4>{});
  if (S <= 8) return pick(std::integral_constant<int, 8>{});
  if (S <= 16) return pick(std::integral_constant<int, 16>{});
  return pick(std::integral_constant<int, 32>{});
}

}  // namespace sf
