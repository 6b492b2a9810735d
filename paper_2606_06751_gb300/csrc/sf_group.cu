// sf_group.cu - the frontier taken within role groups (the App. A role check:
// no global frontier across ranks whose roles differ; Sec. 3 Eq. 1 applied
// inside each group) and reporting-group sums after the frontier (Sec. 3:
// accumulation-indexed stages are aggregated only once the frontier is taken).
//
// group_window_kernel: a CTA walks a contiguous range of steps.  For each
// step its threads stream the rank rows (16-byte loads, two rows in flight,
// the stage prefix in registers) and fold every prefix into a shared-memory
// maximum per (group, stage).  When all 32 lanes of a warp hold ranks of one
// group - the common case of contiguous node groups - the warp first reduces
// each stage in registers and issues one shared atomic; otherwise every lane
// issues its own.  The per-group increments F_g[s] - F_g[s-1] and makespans
// then accumulate in shared memory per window and are added to global memory
// once per window the CTA touches.
//
// group_lanes_kernel: steps of few ranks, one lane per (step, stage).  Three CTA
// barriers and a shared atomic per warp and stage are most of a small step's time
// above; here a warp walks the ranks of 32 / S consecutive steps together, each
// lane keeping the running maximum of the rank's group for its own stage and
// parking it in shared memory when the group changes, so no lane waits for
// another before the step's end.
#include <algorithm>
#include <cmath>
#include <cstdint>
#include <type_traits>

#include <cooperative_groups.h>

#include "sf_device.cuh"
#include "sf_lane_select.cuh"
#include "sf_launch.h"

namespace sf {
namespace {

constexpr int kGrThreads = 256;

struct GroupParams {
  const int64_t* d;
  int64_t T, R, S;
  const int32_t* group;
  int64_t G, t0, W, w_first;
  int64_t* Xg;  // [nW][G][S]
  int64_t* Dg;  // [nW][G]
  uint32_t* status;
};

__device__ __forceinline__ unsigned long long warp_max_u64_all(unsigned long long v) {
  const uint32_t hi = __reduce_max_sync(kFull, static_cast<uint32_t>(v >> 32));
  const uint32_t lo = __reduce_max_sync(kFull, static_cast<uint32_t>(v >> 32) == hi ? static_cast<uint32_t>(v) : 0u);
  return (static_cast<unsigned long long>(hi) << 32) | lo;
}

// One rank row: the stage prefix folded into the group's per-stage maximum.
template <int SC>
__device__ __forceinline__ void fold_row(const GroupParams& p, const int64_t* row, int S, int g, bool valid,
                                         bool warp_uniform, unsigned long long* Fk, uint32_t& dor, uint32_t& tor) {
  constexpr int kCols = SC > 0 ? SC : 1;
  int64_t P = 0;
  if constexpr (SC > 0) {
    int64_t v[kCols];
    if (valid) {
      if constexpr (SC % 2 == 0) {
#pragma unroll
        for (int h = 0; h < SC / 2; ++h) {
          const longlong2 x = __ldg(reinterpret_cast<const longlong2*>(row) + h);
          v[2 * h] = x.x;
          v[2 * h + 1] = x.y;
        }
      } else {
#pragma unroll
        for (int s = 0; s < SC; ++s) v[s] = __ldg(row + s);
      }
    } else {
#pragma unroll
      for (int s = 0; s < SC; ++s) v[s] = 0;
    }
#pragma unroll
    for (int s = 0; s < SC; ++s) {
      dor |= static_cast<uint32_t>(static_cast<uint64_t>(v[s]) >> 32);
      P += v[s];
      if (warp_uniform) {
        const unsigned long long m = warp_max_u64_all(static_cast<unsigned long long>(P));
        if ((threadIdx.x & 31) == 0) atomicMax(&Fk[g * SC + s], m);
      } else if (valid) {
        atomicMax(&Fk[g * SC + s], static_cast<unsigned long long>(P));
      }
    }
  } else {
    for (int s = 0; s < S; ++s) {
      const int64_t v = valid ? __ldg(row + s) : 0;
      dor |= static_cast<uint32_t>(static_cast<uint64_t>(v) >> 32);
      P += v;
      if (warp_uniform) {
        const unsigned long long m = warp_max_u64_all(static_cast<unsigned long long>(P));
        if ((threadIdx.x & 31) == 0) atomicMax(&Fk[g * S + s], m);
      } else if (valid) {
        atomicMax(&Fk[g * S + s], static_cast<unsigned long long>(P));
      }
    }
  }
  tor |= static_cast<uint32_t>(static_cast<uint64_t>(P) >> 32);
}

// Entry i of the step's F_g: the CTA's own, or the largest over the cluster's CTAs.
template <bool SPLIT>
__device__ __forceinline__ int64_t step_frontier(unsigned long long* Fk, int i, int csize, int rank) {
  unsigned long long F = Fk[i];
  if constexpr (SPLIT) {
    for (int c = 1; c < csize; ++c) {
      const int other = rank + c < csize ? rank + c : rank + c - csize;
      const unsigned long long x =
          *cooperative_groups::this_cluster().map_shared_rank(&Fk[i], static_cast<unsigned>(other));
      F = x > F ? x : F;
    }
  }
  return static_cast<int64_t>(F);
}

// Dynamic shared memory: Fk [G][S] u64 (this step's group frontier),
// accX [G][S] i64 and accD [G] i64 (the current window's sums).  SPLIT: a cluster
// of CTAs shares each step's ranks, and its CTAs combine their Fk through
// distributed shared memory, each for every csize-th group.
// Five CTAs per SM: seven and twelve stages would take registers for four, a second
// round for 609 to 760 steps (650 x 2100 x 7 32.8 -> 24.9 us, 650 x 4500 x 12 91 -> 62).
template <int SC, bool SPLIT>
__global__ void __launch_bounds__(kGrThreads, (SPLIT ? SC <= 12 : SC == 7 || SC == 12) ? 5 : 0)
    group_window_kernel(const GroupParams p) {
  namespace cg = cooperative_groups;
  extern __shared__ __align__(16) unsigned char dyn[];
  const int S = SC > 0 ? SC : static_cast<int>(p.S);
  const int G = static_cast<int>(p.G), GS = G * S;
  unsigned long long* Fk = reinterpret_cast<unsigned long long*>(dyn);
  int64_t* accX = reinterpret_cast<int64_t*>(Fk + GS);
  int64_t* accD = accX + GS;
  const int tid = threadIdx.x, lane = tid & 31;
  const int64_t R = p.R;
  int csize = 1, rank = 0;
  if constexpr (SPLIT) {
    csize = static_cast<int>(cg::this_cluster().num_blocks());
    rank = static_cast<int>(cg::this_cluster().block_rank());
  }
  // the CTA's ranks: whole warps, so that a warp's ranks stay those of a node
  const int64_t r_begin = SPLIT ? (R + 31) / 32 * rank / csize * 32 : 0;
  const int64_t r_end = SPLIT ? min(R, (R + 31) / 32 * (rank + 1) / csize * 32) : R;
  const int64_t nb = gridDim.x / csize, b = blockIdx.x / csize;
  const int64_t q = p.T / nb, rr = p.T % nb;
  const int64_t t_begin = q * b + (b < rr ? b : rr), t_end = t_begin + q + (b < rr ? 1 : 0);
  uint32_t dor = 0, tor = 0, bad_group = 0;
  int64_t cur_w = -1;
  int64_t w = 0, w_lo = 0, w_hi = 0;  // steps [w_lo, w_hi) form window w: one division per window

  for (int i = tid; i < GS + G; i += kGrThreads) accX[i] = 0;  // accX and accD are contiguous
  for (int64_t t = t_begin; t < t_end; ++t) {
    if (t < w_lo || t >= w_hi) {
      w = (p.t0 + t) / p.W - p.w_first;
      w_lo = (w + p.w_first) * p.W - p.t0;
      w_hi = w_lo + p.W;
    }
    for (int i = tid; i < GS; i += kGrThreads) Fk[i] = 0;
    if (w != cur_w && cur_w >= 0) {
      // the window changed: add the finished window's sums to global memory
      for (int i = tid; i < GS; i += kGrThreads) {
        if (accX[i]) atomicAdd(reinterpret_cast<unsigned long long*>(&p.Xg[cur_w * GS + i]),
                               static_cast<unsigned long long>(accX[i]));
        accX[i] = 0;
      }
      for (int g = tid; g < G; g += kGrThreads) {
        if (accD[g]) atomicAdd(reinterpret_cast<unsigned long long*>(&p.Dg[cur_w * G + g]),
                               static_cast<unsigned long long>(accD[g]));
        accD[g] = 0;
      }
    }
    cur_w = w;
    __syncthreads();
    const int64_t* dt = p.d + t * R * S;
    constexpr int kRows = (SC > 0 && SC <= 8) ? 2 : 1;
    for (int64_t base = r_begin + tid - lane; base < r_end; base += int64_t(kRows) * kGrThreads) {
      // warp-uniform loop: every lane takes part in the warp reductions
#pragma unroll
      for (int k = 0; k < kRows; ++k) {
        const int64_t r = base + int64_t(k) * kGrThreads + lane;
        const bool in = r < r_end;
        int g = in ? __ldg(p.group + r) : -1;
        const bool ok = g >= 0 && g < G;
        bad_group |= (in && !ok) ? 1u : 0u;
        if (!ok) g = 0;
        const int g0 = __shfl_sync(kFull, g, 0);
        const bool uniform = __all_sync(kFull, ok && g == g0);
        fold_row<SC>(p, dt + (in ? r : 0) * S, S, g, ok, uniform, Fk, dor, tor);
      }
    }
    if constexpr (SPLIT) {
      cg::this_cluster().sync();
    } else {
      __syncthreads();
    }
    // the step's group increments a_g[s] = F_g[s] - F_g[s-1] and makespans
    for (int i = tid; i < GS; i += kGrThreads) {
      const int s = i % S;
      if (SPLIT && i / S % csize != rank) continue;
      const int64_t F = step_frontier<SPLIT>(Fk, i, csize, rank);
      accX[i] += F - (s > 0 ? step_frontier<SPLIT>(Fk, i - 1, csize, rank) : 0);
      if (s == S - 1) accD[i / S] += F;
    }
    if constexpr (SPLIT) {
      cg::this_cluster().sync();  // the others read Fk until here
    } else {
      __syncthreads();
    }
  }
  if (cur_w >= 0) {
    for (int i = tid; i < GS; i += kGrThreads)
      if (accX[i]) atomicAdd(reinterpret_cast<unsigned long long*>(&p.Xg[cur_w * GS + i]),
                             static_cast<unsigned long long>(accX[i]));
    for (int g = tid; g < G; g += kGrThreads)
      if (accD[g]) atomicAdd(reinterpret_cast<unsigned long long*>(&p.Dg[cur_w * G + g]),
                             static_cast<unsigned long long>(accD[g]));
  }
  uint32_t bits = range_bits(__reduce_or_sync(kFull, dor), __reduce_or_sync(kFull, tor));
  if (__any_sync(kFull, bad_group != 0)) bits |= SF_ST_INDEX;
  if (lane == 0) report(p.status, bits);
}

// ---------------------------------------------------------------- few ranks

constexpr int kGlThreads = 128;
constexpr int kGlWarps = kGlThreads / 32;
constexpr int kGlBatch = 8;
constexpr int64_t kGlMaxGroups = 32;
constexpr int64_t kGlMaxRanks = 192;
constexpr int64_t group_lanes_smem(int64_t G) { return kGlWarps * 2 * G * 32 * 8; }  // at most 64 KB

// Whether the lanes take a call, by estimates of both forms' time in us.  A warp's walk
// is a chain of loads and scans per rank, and of one exchange per group at a step's end:
// with few tiles of steps per warp it is slower than a CTA per step (1500 x 128 x 8 in
// node groups 14 us, 41 by lanes).  Fitted to 1866 measured calls of 700 to 100000
// steps, 4 to 192 ranks, 1 to 24 groups (lanes within 10 %, CTAs within 20 %).  Steps
// past 32 bits take the lanes up to twice as long, so they are taken when they are
// half as fast again: then no call of ordinary steps was slower by more than 5 % and 45 of
// 1866 of steps past 32 bits were (at most 1.55 times; all together 2.1 times as fast).
bool use_group_lanes(int64_t T, int64_t R, int64_t S, int64_t G) {
  if (R > kGlMaxRanks || G > kGlMaxGroups) return false;
  const double sms = sm_count();
  const double per_cta = static_cast<double>((T + 32 / S - 1) / (32 / S)) / (sms * kGlWarps);  // tiles, one CTA per SM
  if (per_cta < 1.0) return false;
  const double ctas = static_cast<double>(std::min<int64_t>(5, 227 * 1024 / (group_lanes_smem(G) + 1024)));
  const double rounds = std::ceil(per_cta / ctas);
  const double lanes = 9.0 + rounds * (0.45 + 0.092 * R + 0.53 * G) + per_cta * (0.020 * R + 0.017 * G);
  const double cta = 9.1 + T / (8.0 * sms) * (0.99 + 0.37 * S + 0.018 * G * S + (G > 1 ? 0.126 * S : 0.0));
  return 1.5 * lanes < cta;
}

// Walks the ranks of a warp's steps: park[g][lane] becomes the lane's stage of
// F_g.  32-bit prefixes unless WIDE; returns whether they hold.
template <int LOGS, bool WIDE>
__device__ __forceinline__ bool group_walk(const GroupParams& p, const int64_t* col, int s, uint64_t* park, int lane,
                                           uint32_t& dor, uint32_t& tor, uint32_t& bad_group) {
  using V = std::conditional_t<WIDE, uint64_t, uint32_t>;
  const int R = static_cast<int>(p.R), S = static_cast<int>(p.S), G = static_cast<int>(p.G);
  for (int g = 0; g < G; ++g) park[g * 32 + lane] = 0;
  uint32_t vmax = 0, dhi = 0;
  V best = 0;
  int cur = -1;  // the group `best` belongs to, the same in every lane
  for (int r0 = 0; r0 < R; r0 += kGlBatch) {
    uint2 v[kGlBatch];
    int32_t gr[kGlBatch];
#pragma unroll
    for (int i = 0; i < kGlBatch; ++i) {
      const int r = min(r0 + i, R - 1);  // past the ranks: the last one again, which changes no maximum
      v[i] = load_words(col + int64_t(r) * S);
      gr[i] = __ldg(p.group + r);
    }
#pragma unroll
    for (int i = 0; i < kGlBatch; ++i) {
      const V y = WIDE ? static_cast<V>((static_cast<uint64_t>(v[i].y) << 32) | v[i].x) : static_cast<V>(v[i].x);
      const bool ok = gr[i] >= 0 && gr[i] < G;
      bad_group |= ok ? 0u : 1u;
      V P = ok ? y : V(0);
      if (ok) {
        dhi |= v[i].y;
        vmax = max(vmax, v[i].x);
      }
#pragma unroll
      for (int q = 1; q < (1 << LOGS); q <<= 1) {
        const V up = __shfl_up_sync(kFull, P, q);
        if (s >= q) P += up;
      }
      if constexpr (WIDE)
        if (s == S - 1) tor |= static_cast<uint32_t>(static_cast<uint64_t>(P) >> 32);
      if (ok && gr[i] != cur) {
        if (cur >= 0) park[cur * 32 + lane] = best;
        cur = gr[i];
        best = static_cast<V>(park[cur * 32 + lane]);
      }
      if (ok) best = WIDE ? (static_cast<int64_t>(P) > static_cast<int64_t>(best) ? P : best) : (P > best ? P : best);
    }
  }
  if (cur >= 0) park[cur * 32 + lane] = best;
  if constexpr (WIDE) dor |= dhi;
  uint64_t bound = dhi ? uint64_t(1) << 32 : vmax;  // the lanes' largest values bound the prefixes
#pragma unroll
  for (int q = 1; q < (1 << LOGS); q <<= 1) {
    const uint64_t up = __shfl_up_sync(kFull, bound, q);
    if (s >= q) bound += up;
  }
  return (bound >> 32) == 0;
}

template <int LOGS>
__device__ __noinline__ bool group_walk_wide(const GroupParams& p, const int64_t* col, int s, uint64_t* park, int lane,
                                             uint32_t& dor, uint32_t& tor, uint32_t& bad_group) {
  return group_walk<LOGS, true>(p, col, s, park, lane, dor, tor, bad_group);
}

template <int LOGS>
__global__ void __launch_bounds__(kGlThreads, 5) group_lanes_kernel(const __grid_constant__ GroupParams p) {
  extern __shared__ __align__(16) unsigned char dyn[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int S = static_cast<int>(p.S), G = static_cast<int>(p.G);
  uint64_t* park = reinterpret_cast<uint64_t*>(dyn) + size_t(warp) * 2 * G * 32;  // [G][32]
  int64_t* acc = reinterpret_cast<int64_t*>(park + G * 32);                       // [G][32] the lane's window sums
  const int steps = 32 / S, j = lane / S, s = lane - j * S;
  const int64_t tiles = (p.T + steps - 1) / steps;
  const int64_t nw = int64_t(gridDim.x) * kGlWarps, id = int64_t(blockIdx.x) * kGlWarps + warp;
  const int64_t tile_end = tiles * (id + 1) / nw;
  uint32_t dor = 0, tor = 0, bad_group = 0;
  int64_t w = -1, w_end = 0;  // window of the lane's step: steps below w_end
  bool wide = false;          // walk the next tile in 64 bits at once
  for (int g = 0; g < G; ++g) acc[g * 32 + lane] = 0;
  // The warp's window sums to global memory, those of one window over its steps first
  // (two atomics for every lane and group: 100000 x 128 x 3, 16 groups, 157 -> 115 us).
  auto flush = [&]() {
    const bool one = one_window(w);
    for (int g = 0; g < G; ++g) {
      int64_t x = acc[g * 32 + lane], all;
      acc[g * 32 + lane] = 0;
      if (one) x = sum_steps(x, S, lane);
      all = x;  // the increments of a step add up to its makespan
      if (one)
        for (int o = 1; o < S; o <<= 1) {
          const int64_t up = __shfl_down_sync(kFull, all, o);
          if (lane + o < S) all += up;
        }
      if (w < 0 || (one && lane >= S)) continue;
      if (x != 0)
        atomicAdd(reinterpret_cast<unsigned long long*>(&p.Xg[(w * G + g) * S + s]), static_cast<unsigned long long>(x));
      if (all != 0 && (!one || lane == 0))
        atomicAdd(reinterpret_cast<unsigned long long*>(&p.Dg[w * G + g]), static_cast<unsigned long long>(all));
    }
  };
  for (int64_t tile = tiles * id / nw; tile < tile_end; ++tile) {
    const int64_t t0 = tile * steps;
    const bool live = j < steps && t0 + j < p.T;
    const int64_t t = live ? t0 + j : t0;
    const bool next = live && (w < 0 || t >= w_end);
    if (__any_sync(kFull, next && w >= 0)) flush();
    if (next) {
      w = (p.t0 + t) / p.W - p.w_first;
      w_end = (w + p.w_first + 1) * p.W - p.t0;
    }
    const int64_t* col = p.d + t * p.R * S + s;
    bool fits;
    if (!wide) {
      fits = group_walk<LOGS, false>(p, col, s, park, lane, dor, tor, bad_group);
      wide = !__all_sync(kFull, fits);
      if (wide) group_walk_wide<LOGS>(p, col, s, park, lane, dor, tor, bad_group);
    } else {
      fits = group_walk_wide<LOGS>(p, col, s, park, lane, dor, tor, bad_group);
      wide = !__all_sync(kFull, fits);
    }
    for (int g = 0; g < G; ++g) {
      const int64_t F = static_cast<int64_t>(park[g * 32 + lane]);
      const int64_t before = __shfl_up_sync(kFull, F, 1);
      if (live) acc[g * 32 + lane] += F - (s ? before : 0);
    }
  }
  flush();
  uint32_t bits = range_bits(__reduce_or_sync(kFull, dor), __reduce_or_sync(kFull, tor));
  if (__any_sync(kFull, bad_group != 0)) bits |= SF_ST_INDEX;
  if (lane == 0) report(p.status, bits);
}

template <int LOGS>
cudaError_t launch_group_lanes(const GroupParams& p, cudaStream_t stream) {
  auto kern = group_lanes_kernel<LOGS>;
  const size_t smem = static_cast<size_t>(group_lanes_smem(p.G));
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem));
  int per_sm = 0;
  if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kGlThreads, smem);
  if (e != cudaSuccess) return e;
  const int64_t tiles = (p.T + 32 / p.S - 1) / (32 / p.S);
  const int64_t grid = std::min<int64_t>((tiles + kGlWarps - 1) / kGlWarps, int64_t(sm_count()) * std::max(per_sm, 1));
  count_launch();
  kern<<<static_cast<unsigned>(grid), kGlThreads, smem, stream>>>(p);
  return cudaGetLastError();
}

struct StageGroups {
  int32_t of[32];  // stage -> reporting group
};

__global__ void stage_group_sum_kernel(const int64_t* __restrict__ X, int64_t nW, int S, StageGroups sg, int K,
                                       int64_t* __restrict__ Y) {
  const int64_t n = nW * K;
  for (int64_t i = blockIdx.x * int64_t(blockDim.x) + threadIdx.x; i < n; i += int64_t(gridDim.x) * blockDim.x) {
    const int64_t w = i / K;
    const int k = static_cast<int>(i - w * K);
    int64_t y = 0;
    for (int s = 0; s < S; ++s)
      if (sg.of[s] == k) y += X[w * S + s];
    Y[i] = y;
  }
}

template <int SC>
cudaError_t launch_group_t(const GroupParams& p, size_t smem, cudaStream_t stream) {
  auto kern = group_window_kernel<SC, false>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem));
  if (e != cudaSuccess) return e;
  int per_sm = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kGrThreads, smem) != cudaSuccess || per_sm < 1) {
    cudaGetLastError();
    per_sm = 1;
  }
  count_launch();
  // few steps of many ranks: up to four CTAs per SM, at least 1024 ranks each (us, a
  // CTA per step / split: 1 x 8192 x 8 47 / 16, 100 x 8192 x 8 49 / 25, 250 x 8192 x 8
  // 62 / 41, 100 x 30000 x 16 299 / 130; two CTAs for 1024 ranks, 300 x 1024 x 6 12 / 14;
  // more CTAs, 400 x 2100 x 8 22.6 / 30.8, eight for two, 100 x 9000 x 8 28.5 / 37.8)
  int csize = 1;
  while (csize < 8 && p.T * csize * 2 <= int64_t(sm_count()) * 4 && p.R >= int64_t(csize) * 2048) csize *= 2;
  if (csize > 1) {
    auto split = group_window_kernel<SC, true>;
    e = cudaFuncSetAttribute(split, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem));
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = static_cast<unsigned>(csize);
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.gridDim = dim3(static_cast<unsigned>(p.T * csize));
    cfg.blockDim = dim3(kGrThreads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = stream;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return cudaLaunchKernelEx(&cfg, split, p);
  }
  kern<<<static_cast<unsigned>(std::min(int64_t(per_sm) * sm_count(), p.T)), kGrThreads, smem, stream>>>(p);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_group_windows(const int64_t* d, int64_t T, int64_t R, int64_t S, const int32_t* group, int64_t G,
                                 int64_t t0, int64_t W, int64_t* Xg, int64_t* Dg, uint32_t* status,
                                 cudaStream_t stream) {
  GroupParams p{};
  p.d = d;
  p.T = T;
  p.R = R;
  p.S = S;
  p.group = group;
  p.G = G;
  p.t0 = t0;
  p.W = W;
  p.w_first = t0 / W;
  p.Xg = Xg;
  p.Dg = Dg;
  p.status = status;
  if (use_group_lanes(T, R, S, G)) {
    if (S <= 1) return launch_group_lanes<0>(p, stream);
    if (S <= 2) return launch_group_lanes<1>(p, stream);
    if (S <= 4) return launch_group_lanes<2>(p, stream);
    if (S <= 8) return launch_group_lanes<3>(p, stream);
    if (S <= 16) return launch_group_lanes<4>(p, stream);
    return launch_group_lanes<5>(p, stream);
  }
  const size_t smem = size_t(G) * S * 16 + size_t(G) * 8;
  // Stage counts known to the compiler, whose rows are loaded ahead of their reductions
  // (us, loop over the stages / unrolled: 13421 x 1000 x 5 139 / 115, 10000 x 1024 x 9
  // 184 / 139, 10000 x 700 x 11 174 / 133; 8000 x 1000 x 14 199 / 204).  Up to eight stages
  // a warp takes two rows of 256 ranks, one of them idle in smaller steps (60000 x 200 x 7
  // 233 / 268).
  const bool two_rows = R > kGrThreads;
  switch (S) {
    case 2: if (two_rows) return launch_group_t<2>(p, smem, stream); break;
    case 3: if (two_rows) return launch_group_t<3>(p, smem, stream); break;
    case 5: if (two_rows) return launch_group_t<5>(p, smem, stream); break;
    case 7: if (two_rows) return launch_group_t<7>(p, smem, stream); break;
    case 4: return launch_group_t<4>(p, smem, stream);
    case 6: return launch_group_t<6>(p, smem, stream);
    case 8: return launch_group_t<8>(p, smem, stream);
    case 9: return launch_group_t<9>(p, smem, stream);
    case 10: return launch_group_t<10>(p, smem, stream);
    case 11: return launch_group_t<11>(p, smem, stream);
    case 12: return launch_group_t<12>(p, smem, stream);
    case 16: return launch_group_t<16>(p, smem, stream);
    default: break;
  }
  return launch_group_t<0>(p, smem, stream);
}

cudaError_t launch_stage_group_sum(const int64_t* X, int64_t nW, int64_t S, const int32_t* stage_group, int64_t K,
                                   int64_t* Y, cudaStream_t stream) {
  StageGroups sg{};
  for (int s = 0; s < S; ++s) sg.of[s] = stage_group[s];
  const int64_t n = nW * K;
  const int grid = static_cast<int>(std::max<int64_t>(1, std::min<int64_t>((n + 255) / 256, int64_t(sm_count()) * 8)));
  count_launch();
  stage_group_sum_kernel<<<grid, 256, 0, stream>>>(X, nW, static_cast<int>(S), sg, static_cast<int>(K), Y);
  return cudaGetLastError();
}

}  // namespace sf
