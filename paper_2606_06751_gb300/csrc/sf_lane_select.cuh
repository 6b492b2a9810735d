// sf_lane_select.cuh - kernels that give a lane a (step, stage) or a column: loads,
// sums over a warp's steps, and selection by single lanes, each on a column of up to
// 128 keys that it holds in registers, its loads spread over the warp's 32 columns.
#pragma once

#include "sf_device.cuh"

namespace sf {
namespace {

// Resident CTAs of 128 threads that columns of nmax keys leave registers for,
// and the rows of a column loaded together.
constexpr int lane_ctas(int nmax) { return nmax <= 32 ? 6 : nmax <= 64 ? 4 : nmax <= 104 ? 3 : 2; }
__host__ __device__ constexpr int lane_batch(int nmax) { return nmax == 104 ? 13 : 16; }

// Volatile, so that a batch's loads stay together: hoisted further they would
// hold two registers a row.
__device__ __forceinline__ uint2 load_words(const int64_t* p) {
  uint2 v;
  asm volatile("ld.global.nc.v2.u32 {%0, %1}, [%2];" : "=r"(v.x), "=r"(v.y) : "l"(p));
  return v;
}

// Lanes j S + s hold stage s of a warp's j-th step (0 on lanes past the last whole
// step): the sum over the steps, on lanes s < S.  The whole warp calls it.
__device__ __forceinline__ int64_t sum_steps(int64_t v, int S, int lane) {
  for (int o = S; o < 32; o <<= 1) {
    const int64_t up = __shfl_down_sync(kFull, v, o);
    if (lane + o < 32) v += up;
  }
  return v;
}
__device__ __forceinline__ unsigned __int128 sum_steps(unsigned __int128 v, int S, int lane) {
  uint64_t lo = static_cast<uint64_t>(v), hi = static_cast<uint64_t>(v >> 64);
  for (int o = S; o < 32; o <<= 1) {
    const uint64_t l = __shfl_down_sync(kFull, lo, o), h = __shfl_down_sync(kFull, hi, o);
    if (lane + o < 32) {
      lo += l;
      hi += h + (lo < l ? 1u : 0u);
    }
  }
  return (static_cast<unsigned __int128>(hi) << 64) | lo;
}
// Whether the warp's lanes (w < 0: none yet) are all in the first one's window.
__device__ __forceinline__ bool one_window(int64_t w) {
  const int64_t first = __shfl_sync(kFull, w, 0);
  return __all_sync(kFull, w == first || w < 0);
}

// The kth (from 0) smallest of this lane's n keys (the others hold 0xffffffff),
// which lie in [lo, hi]; the whole warp calls it.  A round counts the keys up to
// a probe, which halves the bracket or, every second round, lies where the
// answer would if the bracket's keys were evenly spread; the lanes' rounds run
// together until every bracket ends at its answer.
template <int N>
__device__ __forceinline__ uint32_t lane_select(const uint32_t (&x)[N], uint32_t n, uint32_t kth, uint32_t lo,
                                                uint32_t hi) {
      // the median is in [lo, hi]; below keys lie under lo, upto at or under hi
      uint32_t below = 0, upto = n;
      for (uint32_t round = 0;; ++round) {
        const bool open = lo < hi && below != kth && upto != kth + 1;
        if (!__any_sync(kFull, open)) break;
        const uint32_t span = hi - lo;
        uint32_t mid = lo + (span >> 1);
        if (round & 1u) {
          const float at = __fdividef(static_cast<float>(kth - below) + 0.5f, static_cast<float>(upto - below));
          mid = lo + min(static_cast<uint32_t>(at * static_cast<float>(span)), span - 1u);
        }
        uint32_t cnt = 0;
#pragma unroll
        for (int i = 0; i < N; ++i) cnt += x[i] <= mid ? 1u : 0u;
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
      // the smallest key from lo on, or the largest up to hi (the smallest of the
      // complements): keys on the other side of the limit wrap to large offsets
      const uint32_t flip = lo == hi || below == kth ? 0u : 0xffffffffu;
      const uint32_t limit = flip ? ~hi : lo;
      uint32_t off = 0xffffffffu;
#pragma unroll
      for (int i = 0; i < N; ++i) off = min(off, (x[i] ^ flip) - limit);
      return (limit + off) ^ flip;
}

}  // namespace
}  // namespace sf
