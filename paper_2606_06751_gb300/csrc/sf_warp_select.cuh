// sf_warp_select.cuh - selection by one warp on a column it holds in registers.
#pragma once

#include "sf_device.cuh"

namespace sf {
namespace {

constexpr int kSelBins = 256;
// Per-warp counters: 256 digit bins, then 48 spare words (a compacted bin of
// at most 32 values and its padding to whole 16-byte groups).  304 words =
// 1216 bytes keeps every warp's block 16-byte aligned.
constexpr int kSelHistWords = kSelBins + 48;

// Shared-memory increment of one counter, issued only when `pred` is set
// (explicitly predicated, so a warp never branches around it).
__device__ __forceinline__ void red_shared_inc_if(uint32_t* counter, bool pred) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %1, 0;\n\t@p red.shared.add.u32 [%0], 1;\n\t}" ::"r"(smem_u32(counter)),
      "r"(static_cast<uint32_t>(pred))
      : "memory");
}

// Radix selection on a column held in registers (x[i] = row lane + 32 i):
// the k-th smallest of the live values, all below 2^nbits.  Padding slots
// must hold 2^nbits - 1: they sort at or after every live value, so counting
// them never moves the rank-k bin and no slot needs a validity test.  The
// first digit is the top 8 bits of the range, [nbits - 8, nbits), so it
// spreads over the 256 bins and its chosen bin usually holds a few percent of
// the column; each later pass counts, predicated, the values that share the
// digits chosen so far.  As soon as the chosen bin holds at most 32 values
// they are compacted into the spare words after the bins (ballot ranks, no
// atomics) and each is ranked by counting.
template <int NPL>
__device__ __forceinline__ uint32_t warp_select_regs(const uint32_t (&x)[NPL], int nbits, uint32_t k,
                                                     uint32_t* hist, int lane) {
  uint32_t prefix = 0, rem = k;
  int hi = nbits;
  bool first = true;
  while (hi > 0) {
    const int sh = hi > 8 ? hi - 8 : 0;
    const uint32_t mask = (1u << (hi - sh)) - 1u;
    reinterpret_cast<uint4*>(hist)[2 * lane] = make_uint4(0, 0, 0, 0);
    reinterpret_cast<uint4*>(hist)[2 * lane + 1] = make_uint4(0, 0, 0, 0);
    __syncwarp();
    if (first) {
#pragma unroll
      for (int i = 0; i < NPL; ++i) atomicAdd(&hist[x[i] >> sh], 1u);  // x < 2^nbits: the bin is below 256
    } else {
#pragma unroll
      for (int i = 0; i < NPL; ++i)
        red_shared_inc_if(&hist[(x[i] >> sh) & mask], (x[i] >> hi) == (prefix >> hi));
    }
    __syncwarp();
    uint32_t digit, below;
    hist_find(hist, rem, lane, digit, below);
    const uint32_t kept = hist[digit];
    rem -= below;
    prefix |= digit << sh;
    hi = sh;
    first = false;
    if (hi > 0 && kept <= 32) {
      uint32_t* cbuf = hist + kSelBins;
      const uint32_t below_lane = (1u << lane) - 1u;
      uint32_t base = 0;
#pragma unroll
      for (int i = 0; i < NPL; ++i) {
        const bool mt = (x[i] >> hi) == (prefix >> hi);
        const uint32_t mm = __ballot_sync(kFull, mt);
        if (mm) {
          if (mt) cbuf[base + __popc(mm & below_lane)] = x[i];
          base += __popc(mm);
        }
      }
      if (lane < 3) cbuf[kept + lane] = 0xffffffffu;  // pad to whole 16-byte groups (kept + 3 <= 35 < 64 spare)
      __syncwarp();
      // rank each bin value by counting (broadcast reads of the bin): the
      // answer is a value with lt <= rem < le.  Padding counts only toward
      // le of the largest key, which no rank below kept can need.
      const uint32_t v = cbuf[lane & 31];
      uint32_t lt = 0, le = 0;
      for (uint32_t q = 0; q < kept; q += 4) {
        const uint4 c = *reinterpret_cast<const uint4*>(cbuf + q);
        lt += (c.x < v) + (c.y < v) + (c.z < v) + (c.w < v);
        le += (c.x <= v) + (c.y <= v) + (c.z <= v) + (c.w <= v);
      }
      const uint32_t hit = __ballot_sync(kFull, static_cast<uint32_t>(lane) < kept && lt <= rem && rem < le);
      const uint32_t ans = __shfl_sync(kFull, v, __ffs(hit) - 1);
      __syncwarp();
      return ans;
    }
    __syncwarp();
  }
  return prefix;
}

// The k-th smallest (from 0) of the n live values x[i] in [0, hi]; padding slots
// hold hi or more.  A round counts the values up to a probe (one redux), which
// halves the bracket or, every second round, lies where the answer would if the
// bracket's values were evenly spread.  Outliers that stretch the range cost it a
// few rounds, where they cost the histogram's first pass most of its bins.
template <int NPL>
__device__ __forceinline__ uint32_t warp_bisect_regs(const uint32_t (&x)[NPL], uint32_t n, uint32_t k, uint32_t hi) {
  uint32_t lo = 0, below = 0, upto = n;
  for (uint32_t round = 0; lo < hi && below != k && upto != k + 1; ++round) {
    const uint32_t span = hi - lo;
    uint32_t mid = lo + (span >> 1);
    if (round & 1u) {
      const float at = __fdividef(static_cast<float>(k - below) + 0.5f, static_cast<float>(upto - below));
      mid = lo + min(static_cast<uint32_t>(at * static_cast<float>(span)), span - 1u);
    }
    uint32_t c = 0;
#pragma unroll
    for (int i = 0; i < NPL; ++i) c += x[i] <= mid ? 1u : 0u;
    c = __reduce_add_sync(kFull, c);
    if (c > k) {
      hi = mid;
      upto = c;
    } else {
      lo = mid + 1;
      below = c;
    }
  }
  if (lo == hi) return lo;
  const uint32_t flip = below == k ? 0u : 0xffffffffu;
  const uint32_t limit = flip ? ~hi : lo;
  uint32_t off = 0xffffffffu;
#pragma unroll
  for (int i = 0; i < NPL; ++i) off = min(off, (x[i] ^ flip) - limit);
  off = __reduce_min_sync(kFull, off);
  return (limit + off) ^ flip;
}

}  // namespace
}  // namespace sf
