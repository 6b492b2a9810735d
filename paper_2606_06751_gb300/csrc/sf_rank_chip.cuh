// sf_rank_chip.cuh - shared by the on-chip rank statistics (sf_rank_lanes.cu and
// sf_rank_chip.cu): parameters, device pieces and the launch.
#pragma once

#include <algorithm>
#include <cstdint>

#include "sf_device.cuh"
#include "sf_launch.h"

namespace sf {

struct ChipParams {
  const int64_t* d;
  int64_t T;
  int R, S;
  int of_prefix;  // 1: order statistics of P (lag); 0: of d (spread)
  int64_t t0, W, w_first;
  int64_t *L, *dL, *G;  // [T][S], nullable
  int64_t *Lw, *Gw;     // [nW][S] window sums, nullable
  int64_t* spread;      // [nW][S], nullable
  uint32_t* status;
  int ld;   // key column stride in words (rank_step_kernel)
  int wpc;  // warps per column (rank_step_kernel)
};

// Steps of few ranks: a lane per column.
constexpr int kRankLaneMax = 128;
cudaError_t launch_rank_lanes(const ChipParams& p, cudaStream_t stream);
// ... or a warp per step (65 to 128 ranks, up to 8 stages).
constexpr int kRankWarpMin = 65, kRankWarpMaxS = 8;
cudaError_t launch_rank_warp(const ChipParams& p, cudaStream_t stream);

namespace {

constexpr uint32_t kSign32 = 0x80000000u;
constexpr int kChipMaxS = 32;


__device__ __forceinline__ uint32_t hi32(int64_t v) {
  return static_cast<uint32_t>(static_cast<uint64_t>(v) >> 32);
}

// The two largest of (a1 >= a2) and x; an equal value counts as the second.
__device__ __forceinline__ void top2_add(uint32_t& a1, uint32_t& a2, uint32_t x) {
  a2 = max(a2, min(a1, x));
  a1 = max(a1, x);
}

// The warp's two largest from each lane's.
__device__ __forceinline__ void warp_top2(uint32_t& a1, uint32_t& a2) {
  const uint32_t m = __reduce_max_sync(kFull, a1);
  const bool at = a1 == m;
  const uint32_t s = __reduce_max_sync(kFull, at ? a2 : a1);
  a2 = __popc(__ballot_sync(kFull, at)) > 1 ? m : s;
  a1 = m;
}

// Value of (rank r, stage s) of a step, read from d.
__device__ __forceinline__ int64_t step_value(const int64_t* dt, int S, bool of_prefix, int r, int s) {
  const int64_t* row = dt + int64_t(r) * S;
  if (!of_prefix) return __ldg(row + s);
  int64_t P = 0;
#pragma unroll 1
  for (int i = 0; i <= s; ++i) P += __ldg(row + i);
  return P;
}

// True if a value of rows r0, r0 + stride, ... lies 2^31 or more from rank 0's
// (ref, in shared memory).
__device__ __noinline__ bool far_from_first(const int64_t* dt, int R, int S, bool of_prefix, const int64_t* ref, int r0,
                                            int stride) {
  bool bad = false;
#pragma unroll 1
  for (int r = r0; r < R; r += stride) {
    const int64_t* row = dt + int64_t(r) * S;
    int64_t x = 0;
#pragma unroll 4
    for (int s = 0; s < S; ++s) {
      const int64_t v = __ldg(row + s);
      x = of_prefix ? x + v : v;
      bad |= (static_cast<uint64_t>(x - ref[s] + 0x80000000ll) >> 32) != 0;
    }
  }
  return bad;
}

// One column of R 64-bit values in shared memory, by one warp: radix
// selection, one byte of the range per pass.  hist: 256 counters of this warp.
__device__ __noinline__ void column_64(const int64_t* col, int R, uint32_t* hist, int lane, int64_t& med, int64_t& top,
                                       int64_t& second) {
  constexpr uint64_t kSign = 1ull << 63;
  auto key = [&](int r) { return static_cast<uint64_t>(col[r]) ^ kSign; };
  uint64_t lo = ~0ull, a1 = 0, a2 = 0;
#pragma unroll 1
  for (int r = lane; r < R; r += 32) {
    const uint64_t x = key(r);
    lo = x < lo ? x : lo;
    const uint64_t less = x < a1 ? x : a1;
    a2 = less > a2 ? less : a2;
    a1 = x > a1 ? x : a1;
  }
  lo = warp_min_u64(lo);
  const uint64_t m = warp_max_u64(a1);
  const uint64_t s2 = warp_max_u64(a1 == m ? a2 : a1);
  a2 = __popc(__ballot_sync(kFull, a1 == m)) > 1 ? m : s2;
  const uint64_t range = m - lo;
  const int bytes = range ? (71 - __clzll(static_cast<long long>(range))) / 8 : 0;
  uint64_t pref = 0;
  uint32_t rem = static_cast<uint32_t>((R - 1) / 2);
#pragma unroll 1
  for (int b = bytes - 1; b >= 0; --b) {
    const int shift = 8 * b;
#pragma unroll
    for (int i = 0; i < 8; ++i) hist[lane + 32 * i] = 0;
    __syncwarp();
#pragma unroll 2
    for (int r = lane; r < R; r += 32) {
      const uint64_t off = key(r) - lo;
      if (shift == 56 || (off >> (shift + 8)) == (pref >> (shift + 8)))
        atomicAdd(&hist[static_cast<uint32_t>(off >> shift) & 255u], 1u);
    }
    __syncwarp();
    uint32_t digit, below;
    hist_find(hist, rem, lane, digit, below);
    rem -= below;
    pref |= static_cast<uint64_t>(digit) << shift;
    __syncwarp();
  }
  med = static_cast<int64_t>((lo + pref) ^ kSign);
  top = static_cast<int64_t>(m ^ kSign);
  second = static_cast<int64_t>((R >= 2 ? a2 : m) ^ kSign);
}

// 64-bit values of stages [s0, s1) of every rank of a step, read again from d
// into shared memory: stage s at col + (s - s0) ld.  The whole CTA calls it.
__device__ __noinline__ void columns_to_smem(const int64_t* dt, int R, int S, bool of_prefix, int s0, int s1,
                                             int64_t* col, int ld) {
#pragma unroll 1
  for (int r = threadIdx.x; r < R; r += blockDim.x) {
    const int64_t* row = dt + int64_t(r) * S;
    int64_t x = 0;
#pragma unroll 4
    for (int s = 0; s < s1; ++s) {
      const int64_t v = __ldg(row + s);
      x = of_prefix ? x + v : v;
      if (s >= s0) col[(s - s0) * ld + r] = x;
    }
  }
}

// Starts the copy of a step (its whole 16-byte groups) into L2.  One thread.
__device__ __forceinline__ void prefetch_step(const int64_t* dt, int64_t values) {
  const uint64_t a = reinterpret_cast<uint64_t>(dt) & ~15ull, e = reinterpret_cast<uint64_t>(dt + values) & ~15ull;
  if (e > a)
    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(a), "r"(static_cast<uint32_t>(e - a)) : "memory");
}

// Adds `v` to a window sum.
__device__ __forceinline__ void add_window(int64_t* sums, int64_t at, int64_t v) {
  if (v) atomicAdd(reinterpret_cast<unsigned long long*>(sums + at), static_cast<unsigned long long>(v));
}

template <typename K>
cudaError_t launch_chip(K kern, const ChipParams& p, int threads, size_t smem, int64_t per_cta, cudaStream_t stream) {
  if (smem > 48 * 1024) {
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem));
    if (e != cudaSuccess) return e;
  }
  int per_sm = 0;
  const cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, threads, smem);
  if (e != cudaSuccess) return e;
  const int64_t grid = std::min<int64_t>((p.T + per_cta - 1) / per_cta, int64_t(sm_count()) * std::max(per_sm, 1));
  count_launch();
  kern<<<static_cast<unsigned>(grid), threads, smem, stream>>>(p);
  return cudaGetLastError();
}

}  // namespace
}  // namespace sf
