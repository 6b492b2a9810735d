// sf_rank_chip.cu - cross-rank order statistics per (step, stage) for steps
// that fit one SM: the lower median over ranks of the prefixes P[t,r,s] (lag)
// or of the durations (raw rank spread), the maximum and the second largest
// value.  d is read once and nothing is written but the results; sf_rank.cu
// takes the larger steps through a scratch in L2.
//
// Which kernel takes a call (rank_form), and what each measured as lag over 0.1 to
// 4.1 GB against the passes through L2 (whose per-column CTAs have little to do on few
// ranks):
//  rank_lanes_kernel (sf_rank_lanes.cu) - up to 128 ranks: one lane per column,
//    its keys in registers (100000 x 16 x 8 3133 -> 44 us, 131072 x 64 x 16
//    7850 -> 391 us).
//  rank_warp_kernel (sf_rank_warp.cu) - 65 to 128 ranks with up to 8 stages: one
//    warp per step, lane l holding ranks l, l + 32, ..., all stages; the S
//    medians are searched together by counting (one redux per column and
//    round).  The lanes form's columns leave room for eight warps per SM there
//    (100000 x 128 x 8: 3207 us through L2, 431 us by lanes, 250 us).
//  rank_column_kernel - one CTA per step of up to 2048 ranks, the keys
//    transposed through shared memory (a column of ranks per stage); a warp
//    then holds a column in registers and searches it by a radix selection, 8
//    bits a pass, or by counting.  Bound by the chain of loads, barrier and
//    selection, which resident CTAs overlap (50000 x 1024 x 10: 3567 -> 1118 us,
//    60000 x 256 x 8 442 us).  It also takes few steps of up to 128 ranks.
//  rank_step_kernel - the same for more ranks, one to eight warps per column
//    reading the keys from shared memory in each pass (10000 x 4000 x 3:
//    1247 -> 492 us; with eight stages it would be as slow as the passes
//    through L2: 600 x 2500 x 8 56 / 60 us, of long steps 62 / 83).
//
// Keys are the values' low words.  A step whose values all fit 32 bits (rank
// totals below 4.29 s) orders by them as they are; otherwise the step is read
// again and keys are taken relative to rank 0's value, exact while no value is
// 2^31 or more away from it; a step where one is selects on 64-bit values.
#include "sf_bracket.h"
#include "sf_rank_chip.cuh"
#include "sf_warp_select.cuh"

namespace sf {
namespace {

// ---------------------------------------------------------------- CTA per step, columns in registers

constexpr int kColThreads = 256;
constexpr int kColMaxRanks = 2048;

// NPL >= ceil(R / 32); VEC: S even, rows read 16 bytes at a time.
template <int NPL, bool VEC>
__global__ void __launch_bounds__(kColThreads, NPL <= 32 ? 3 : 2) rank_column_kernel(const ChipParams p) {
  extern __shared__ __align__(16) uint32_t smem[];
  __shared__ int64_t sref[kChipMaxS], slag[kChipMaxS];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, threads = blockDim.x, warps = threads >> 5;
  const int S = p.S, R = p.R, ld = p.ld;
  uint32_t* hist = smem + warp * kSelHistWords;
  uint32_t* keys = smem + warps * kSelHistWords;  // [S][ld]
  const uint32_t kth = static_cast<uint32_t>((R - 1) / 2);
  const bool gaps = p.G || p.Gw;
  uint32_t dor = 0, tor = 0;
  for (int64_t t = blockIdx.x; t < p.T; t += gridDim.x) {
    const int64_t* dt = p.d + t * R * S;
    uint32_t wide = 0;
    for (int r = tid; r < R; r += threads) {
      const int64_t* row = dt + int64_t(r) * S;
      uint32_t* out = keys + r;
      uint64_t P = 0;
      uint32_t vh = 0;
      auto take = [&](int64_t v, int s) {
        vh |= hi32(v);
        P += static_cast<uint64_t>(v);
        out[s * ld] = p.of_prefix ? static_cast<uint32_t>(P) : static_cast<uint32_t>(v);
      };
      if constexpr (VEC) {
        // four 16-byte loads in flight
        int s = 0;
        for (; s + 8 <= S; s += 8) {
          longlong2 x[4];
#pragma unroll
          for (int h = 0; h < 4; ++h) x[h] = __ldg(reinterpret_cast<const longlong2*>(row + s) + h);
#pragma unroll
          for (int h = 0; h < 4; ++h) {
            take(x[h].x, s + 2 * h);
            take(x[h].y, s + 2 * h + 1);
          }
        }
#pragma unroll 3
        for (; s < S; s += 2) {
          const longlong2 x = __ldg(reinterpret_cast<const longlong2*>(row + s));
          take(x.x, s);
          take(x.y, s + 1);
        }
      } else {
#pragma unroll 4
        for (int s = 0; s < S; ++s) take(__ldg(row + s), s);
      }
      dor |= vh;
      const uint32_t th = static_cast<uint32_t>(P >> 32);
      tor |= th;
      wide |= vh | (p.of_prefix ? th : 0u);
    }
    const bool rel = __syncthreads_or(wide != 0) != 0;
    if (tid == 0 && t + gridDim.x < p.T) prefetch_step(dt + int64_t(gridDim.x) * R * S, int64_t(R) * S);
    bool far = false;
    if (rel) {
      if (tid < S) sref[tid] = step_value(dt, S, p.of_prefix, 0, tid);
      __syncthreads();
      far = __syncthreads_or(far_from_first(dt, R, S, p.of_prefix, sref, tid, threads)) != 0;
    }
    auto emit = [&](int s, int64_t med, int64_t top, int64_t second) {  // one thread per column
      const int64_t lag = top - med, gap = top - second;
      slag[s] = lag;
      if (p.L) p.L[t * S + s] = lag;
      if (p.G) p.G[t * S + s] = gap;
      if (p.Lw || p.Gw || p.spread) {
        const int64_t at = ((p.t0 + t) / p.W - p.w_first) * S + s;
        if (p.Lw) add_window(p.Lw, at, lag);
        if (p.Gw) add_window(p.Gw, at, gap);
        if (p.spread) add_window(p.spread, at, lag);
      }
    };
    if (far) {  // 64-bit values, half of the stages at a time
      const int part = max(S, 2) / 2;
      int64_t* col = reinterpret_cast<int64_t*>(keys);
      for (int s0 = 0; s0 < S; s0 += part) {
        const int s1 = min(s0 + part, S);
        __syncthreads();
        columns_to_smem(dt, R, S, p.of_prefix, s0, s1, col, ld);
        __syncthreads();
        for (int s = s0 + warp; s < s1; s += warps) {
          int64_t med, top, second;
          column_64(col + (s - s0) * ld, R, hist, lane, med, top, second);
          if (lane == 0) emit(s, med, top, second);
          __syncwarp();
        }
      }
    } else {
      for (int s = warp; s < S; s += warps) {
        int64_t med, top, second;
        const int64_t ref = rel ? sref[s] : 0;
        const uint32_t bias = rel ? static_cast<uint32_t>(ref) - kSign32 : 0u;
        const uint32_t* col = keys + s * ld;
        uint32_t x[NPL];
        uint32_t mn = 0xffffffffu, k1 = 0, k2 = 0;
        // slots of the lower half always hold a rank (R > 16 NPL) but for the smallest form
        auto live = [&](int i) { return (NPL > 8 && i < NPL / 2) || lane + 32 * i < R; };
#pragma unroll
        for (int i = 0; i < NPL; ++i) x[i] = live(i) ? col[lane + 32 * i] - bias : 0xffffffffu;
#pragma unroll
        for (int i = 0; i < NPL; i += 2) {
          mn = __vimin3_u32(mn, x[i], x[i + 1]);
          const uint32_t u = live(i) ? x[i] : 0u, v = live(i + 1) ? x[i + 1] : 0u;
          if (gaps) {
            const uint32_t big = max(u, v);
            k2 = __vimax3_u32(k2, min(u, v), min(k1, big));
            k1 = max(k1, big);
          } else {
            k1 = __vimax3_u32(k1, u, v);
          }
        }
        // Between the largest of the lanes' minima and the smallest of their maxima
        // lie the middle three quarters of a column without its outliers.  Where
        // outliers stretch the range over that more than fourfold they would crowd
        // the column into a few bins: it is bisected instead (1024 x 10 lag with 0.5 %
        // of the cells heavy-tailed: 1312 against 1499 us; without, 1195 against
        // 1118 us).  So are columns of up to 512 ranks, too short to repay a
        // histogram (512 x 12: 308 against 342 us).
        const uint32_t A = __reduce_max_sync(kFull, mn), B = __reduce_min_sync(kFull, k1);
        mn = __reduce_min_sync(kFull, mn);
        if (gaps) warp_top2(k1, k2);
        else k1 = __reduce_max_sync(kFull, k1);
        const uint32_t range = k1 - mn;
        uint32_t ans = mn;
        if (range != 0) {
          const int nbits = 32 - __clz(static_cast<int>(range));
          const uint32_t pad = nbits == 32 ? 0xffffffffu : (1u << nbits) - 1u;  // sorts at or after every key
#pragma unroll
          for (int i = 0; i < NPL; ++i) x[i] = live(i) ? x[i] - mn : pad;
          if (NPL <= 16 || A >= B || B - A < (range >> 2))
            ans += warp_bisect_regs<NPL>(x, static_cast<uint32_t>(R), kth, range);
          else
            ans += warp_select_regs<NPL>(x, nbits, kth, hist, lane);
        }
        if (R < 2) k2 = k1;
        auto value = [&](uint32_t key) {
          return rel ? ref + static_cast<int64_t>(static_cast<int32_t>(key ^ kSign32)) : static_cast<int64_t>(key);
        };
        med = value(ans);
        top = value(k1);
        second = value(k2);
        if (lane == 0) emit(s, med, top, second);
        __syncwarp();
      }
    }
    __syncthreads();  // the columns have been read, the lags are written
    if (p.dL && tid < S) p.dL[t * S + tid] = slag[tid] - (tid ? slag[tid - 1] : 0);
    // slag is next written after the next step's first __syncthreads_or
  }
  const uint32_t bits = range_bits(__reduce_or_sync(kFull, dor), p.of_prefix ? __reduce_or_sync(kFull, tor) : 0u);
  if (lane == 0) report(p.status, bits);
}

// ---------------------------------------------------------------- CTA per step, columns in shared memory

constexpr int kStepWarps = 16;
constexpr int kStepThreads = kStepWarps * 32;
constexpr int kColWords = 256 + 48 + 6 * 8;  // per column group: bins, gathered keys, their count, warp partials

template <int SMAX, bool VEC>
__global__ void __launch_bounds__(kStepThreads, 2) rank_step_kernel(const ChipParams p) {
  constexpr int U = SMAX <= 8 ? 2 : 1;  // rank rows in flight per thread
  extern __shared__ __align__(16) uint32_t smem[];
  __shared__ int64_t sref[kChipMaxS], slag[kChipMaxS];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int S = p.S, R = p.R, ld = p.ld;
  uint32_t* keys = smem;  // [S][ld]
  const int wpc = p.wpc, ngroups = kStepWarps / wpc;
  const int group = warp / wpc, gl = tid - group * wpc * 32, gn = wpc * 32;  // column group, thread within it
  uint32_t* hist = smem + max(S, 2) * ld + group * kColWords;
  uint32_t* cbuf = hist + 256;          // 48 words
  uint32_t* ncand = hist + 256 + 36;    // past the 32 keys and their padding
  uint32_t* part = hist + 256 + 48;     // [6][8] per-warp minimum, maximum, second, bracket, keys outside it
  auto group_sync = [&]() {
    if (wpc == 1) __syncwarp();
    else named_barrier(static_cast<uint32_t>(1 + group), static_cast<uint32_t>(gn));
  };
  const uint32_t kth = static_cast<uint32_t>((R - 1) / 2);
  uint32_t dor = 0, tor = 0;
  for (int64_t t = blockIdx.x; t < p.T; t += gridDim.x) {
    const int64_t* dt = p.d + t * R * S;
    uint32_t wide = 0;
    for (int r0 = tid; r0 < R; r0 += kStepThreads * U) {
      int64_t v[U][SMAX];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int r = r0 + u * kStepThreads;
        if (r >= R) break;
        const int64_t* row = dt + int64_t(r) * S;
        if constexpr (VEC) {
#pragma unroll
          for (int s = 0; s < SMAX; s += 2) {
            if (s >= S) break;
            const longlong2 x = __ldg(reinterpret_cast<const longlong2*>(row + s));
            v[u][s] = x.x;
            v[u][s + 1] = x.y;
          }
        } else {
#pragma unroll
          for (int s = 0; s < SMAX; ++s) {
            if (s >= S) break;
            v[u][s] = __ldg(row + s);
          }
        }
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int r = r0 + u * kStepThreads;
        if (r >= R) break;
        uint64_t P = 0;
        uint32_t vh = 0;
#pragma unroll
        for (int s = 0; s < SMAX; ++s) {
          if (s >= S) break;
          vh |= hi32(v[u][s]);
          P += static_cast<uint64_t>(v[u][s]);
          keys[s * ld + r] = p.of_prefix ? static_cast<uint32_t>(P) : static_cast<uint32_t>(v[u][s]);
        }
        dor |= vh;
        const uint32_t th = static_cast<uint32_t>(P >> 32);
        tor |= th;
        wide |= vh | (p.of_prefix ? th : 0u);
      }
    }
    const bool rel = __syncthreads_or(wide != 0) != 0;
    if (tid == 0 && t + gridDim.x < p.T) prefetch_step(dt + int64_t(gridDim.x) * R * S, int64_t(R) * S);
    bool far = false;
    if (rel) {
      if (tid < S) sref[tid] = step_value(dt, S, p.of_prefix, 0, tid);
      __syncthreads();
      far = __syncthreads_or(far_from_first(dt, R, S, p.of_prefix, sref, tid, kStepThreads)) != 0;
    }
    auto emit = [&](int s, int64_t med, int64_t top, int64_t second) {  // one thread per column
      const int64_t lag = top - med, gap = top - second;
      slag[s] = lag;
      if (p.L) p.L[t * S + s] = lag;
      if (p.G) p.G[t * S + s] = gap;
      if (p.Lw || p.Gw || p.spread) {
        const int64_t at = ((p.t0 + t) / p.W - p.w_first) * S + s;
        if (p.Lw) add_window(p.Lw, at, lag);
        if (p.Gw) add_window(p.Gw, at, gap);
        if (p.spread) add_window(p.spread, at, lag);
      }
    };
    if (far) {  // 64-bit values, half of the stages at a time, a warp of each group
      const int part = max(S, 2) / 2;
      int64_t* col = reinterpret_cast<int64_t*>(keys);
      for (int s0 = 0; s0 < S; s0 += part) {
        const int s1 = min(s0 + part, S);
        __syncthreads();
        columns_to_smem(dt, R, S, p.of_prefix, s0, s1, col, ld);
        __syncthreads();
        if (gl < 32)
          for (int s = s0 + group; s < s1; s += ngroups) {
            int64_t med, top, second;
            column_64(col + (s - s0) * ld, R, hist, lane, med, top, second);
            if (lane == 0) emit(s, med, top, second);
            __syncwarp();
          }
      }
    } else {
      for (int s = group; s < S; s += ngroups) {
        int64_t med, top, second;
        const int64_t ref = rel ? sref[s] : 0;
        const uint32_t bias = rel ? static_cast<uint32_t>(ref) - kSign32 : 0u;
        const uint32_t* col = keys + s * ld;
        const uint4* col4 = reinterpret_cast<const uint4*>(col);
        const int nq = R >> 2;
        // every key of the column, four to a load
        auto each = [&](auto f) {
#pragma unroll 2
          for (int i = gl; i < nq; i += gn) {
            const uint4 x = col4[i];
            f(x.x - bias);
            f(x.y - bias);
            f(x.z - bias);
            f(x.w - bias);
          }
          for (int r = 4 * nq + gl; r < R; r += gn) f(col[r] - bias);
        };
        uint32_t lo = 0xffffffffu, k1 = 0, k2 = 0;
        each([&](uint32_t x) {
          lo = min(lo, x);
          top2_add(k1, k2, x);
        });
        // A first bracket around the median: between the largest of the lanes'
        // minima and the smallest of their maxima, lanes merged until each
        // stands for 16 keys or more.  It keeps the middle three quarters of a
        // column and leaves its outliers out; a median outside it costs one
        // more pass.
        uint32_t A = lo, B = k1;
        for (int o = 1; o < 32 && R * o < 16 * gn; o <<= 1) {
          A = min(A, __shfl_xor_sync(kFull, A, o));
          B = max(B, __shfl_xor_sync(kFull, B, o));
        }
        A = __reduce_max_sync(kFull, A);
        B = __reduce_min_sync(kFull, B);
        lo = __reduce_min_sync(kFull, lo);
        warp_top2(k1, k2);
        if (wpc > 1) {
          const int me = gl >> 5;
          if (lane == 0) {
            part[me] = lo;
            part[8 + me] = k1;
            part[16 + me] = k2;
            part[24 + me] = A;
            part[32 + me] = B;
          }
          group_sync();
          lo = part[0];
          k1 = part[8];
          k2 = part[16];
          A = part[24];
          B = part[32];
          for (int q = 1; q < wpc; ++q) {
            lo = min(lo, part[q]);
            const uint32_t b1 = part[8 + q], b2 = part[16 + q];
            k2 = max(min(k1, b1), max(k2, b2));
            k1 = max(k1, b1);
            A = min(A, part[24 + q]);
            B = max(B, part[32 + q]);
          }
        }
        if (A > B) {
          A = lo;
          B = k1;
        }
        // the median is the rem-th key (from 0) of those in the bracket
        KeyBracket br = KeyBracket::between(A, B);
        uint32_t rem = kth, ans = lo;
        bool first = true;
        for (int round = 0; lo != k1 && round < kBracketRounds; ++round) {
          const int sh = br.shift();
          for (int i = gl; i < 64; i += gn) reinterpret_cast<uint4*>(hist)[i] = make_uint4(0, 0, 0, 0);
          if (gl == 0) *ncand = 0;
          group_sync();
          if (first) {
            uint32_t out = 0;  // keys below the bracket in the low half word, above it in the high one
            each([&](uint32_t x) {
              const uint32_t o = x - br.lo;
              red_shared_inc_if(&hist[(o >> sh) & 255u], o <= br.span);
              out += o <= br.span ? 0u : x < br.lo ? 1u : 0x10000u;
            });
            out = __reduce_add_sync(kFull, out);
            if (lane == 0) part[40 + (gl >> 5)] = out;
          } else {
            each([&](uint32_t x) {
              const uint32_t o = x - br.lo;
              red_shared_inc_if(&hist[(o >> sh) & 255u], o <= br.span);
            });
          }
          group_sync();
          if (first) {
            first = false;
            uint32_t out = 0;
            for (int q = 0; q < wpc; ++q) out += part[40 + q];
            const uint32_t below = out & 0xffffu, upto = static_cast<uint32_t>(R) - (out >> 16);
            if (kth < below || kth >= upto) {  // outside the bracket
              if (kth < below) {
                br = KeyBracket::between(lo, br.lo - 1);
              } else {
                br = KeyBracket::between(br.last() + 1, k1);
                rem = kth - upto;
              }
              group_sync();  // every warp has read the counts
              continue;
            }
            rem = kth - below;
          }
          uint32_t digit, less;
          hist_find(hist, rem, lane, digit, less);
          const uint32_t kept = hist[digit];
          rem -= less;
          br.narrow(digit);
          ans = br.lo;
          if (sh == 0) break;
          if (kept <= 32) {
            each([&](uint32_t x) {
              if (br.has(x)) cbuf[atomicAdd(ncand, 1u) & 31u] = x;
            });
            group_sync();
            const uint32_t v = static_cast<uint32_t>(lane) < kept ? cbuf[lane] : 0xffffffffu;
            uint32_t lt = 0, le = 0;
            for (uint32_t q = 0; q < kept; ++q) {
              const uint32_t c = __shfl_sync(kFull, v, static_cast<int>(q));
              lt += c < v ? 1u : 0u;
              le += c <= v ? 1u : 0u;
            }
            const uint32_t hit = __ballot_sync(kFull, static_cast<uint32_t>(lane) < kept && lt <= rem && rem < le);
            ans = __shfl_sync(kFull, v, __ffs(hit) - 1);
            break;
          }
          group_sync();  // the bins have been read
        }
        group_sync();  // the group's words are free for its next column
        if (R < 2) k2 = k1;
        auto value = [&](uint32_t key) {
          return rel ? ref + static_cast<int64_t>(static_cast<int32_t>(key ^ kSign32)) : static_cast<int64_t>(key);
        };
        med = value(ans);
        top = value(k1);
        second = value(k2);
        if (gl == 0) emit(s, med, top, second);
      }
    }
    __syncthreads();  // the columns have been read, the lags are written
    if (p.dL && tid < S) p.dL[t * S + tid] = slag[tid] - (tid ? slag[tid - 1] : 0);
    // slag is next written after the next step's first __syncthreads_or
  }
  const uint32_t bits = range_bits(__reduce_or_sync(kFull, dor), p.of_prefix ? __reduce_or_sync(kFull, tor) : 0u);
  if (lane == 0) report(p.status, bits);
}

// ---------------------------------------------------------------- host side

size_t step_smem(int64_t R, int64_t S) {
  const int64_t ld = (R + 3) & ~int64_t(3);
  return size_t(std::max<int64_t>(S, 2)) * ld * 4 + size_t(kStepWarps) * kColWords * 4;
}

constexpr size_t kStepSmemMax = 112 * 1024;  // two CTAs per SM

// rank_column_kernel: the fewest warps that take the columns in as few rounds as eight would
int column_warps(int64_t S) {
  const int64_t rounds = (S + 7) / 8;
  return static_cast<int>((S + rounds - 1) / rounds);
}

size_t column_smem(int64_t R, int64_t S) {
  const int64_t ld = (R + 3) & ~int64_t(3);
  return size_t(std::max<int64_t>(S, 2)) * ld * 4 + size_t(column_warps(S)) * kSelHistWords * 4;
}

template <int SMAX>
cudaError_t launch_step(ChipParams p, cudaStream_t stream) {
  p.ld = (p.R + 3) & ~3;
  // warps per column: as many as keep every column in one round and give each at least 256 keys
  p.wpc = 1;
  while (p.wpc < 8 && 2 * p.wpc * p.S <= kStepWarps && p.R >= 512 * p.wpc) p.wpc *= 2;
  const size_t smem = step_smem(p.R, p.S);
  return p.S % 2 == 0 ? launch_chip(rank_step_kernel<SMAX, true>, p, kStepThreads, smem, 1, stream)
                      : launch_chip(rank_step_kernel<SMAX, false>, p, kStepThreads, smem, 1, stream);
}

template <int NPL>
cudaError_t launch_column(ChipParams p, cudaStream_t stream) {
  p.ld = (p.R + 3) & ~3;
  const int threads = column_warps(p.S) * 32;
  const size_t smem = column_smem(p.R, p.S);
  return p.S % 2 == 0 ? launch_chip(rank_column_kernel<NPL, true>, p, threads, smem, 1, stream)
                      : launch_chip(rank_column_kernel<NPL, false>, p, threads, smem, 1, stream);
}

// The form of a call's steps.  The lines, with lag in us, also of steps 64 times as long
// (in brackets), through L2 / by the form the line is drawn against / by the form chosen:
//  - Few steps of up to 128 ranks leave the lanes a tile or two per warp, and one past 32
//    bits, which its warp takes again column by column, waits for nothing else: a CTA per
//    step up to 10 steps per SM (300 x 64 x 4 14.4 / 10.3 / 6.2 (16.5 / 75.8 / 8.3),
//    1500 x 64 x 8 57.9 / 10.3 / 12.3 (58.7 / 76.9 / 16.4)).  Columns enough for the lanes
//    come from fewer steps of many stages, and a column of 16 ranks is short (column form /
//    lanes 1300 x 16 x 16 16 / 6.2 (21 / 68), 855 x 15 x 32 18.5 / 6.2 (37 / 72),
//    855 x 60 x 32 23 / 12 (54 / 101), 855 x 96 x 24 18 / 16 (43 / 83)).
//  - The column form has a warp per stage, too few to load few steps of many ranks and few
//    stages: those take the step form (40 x 1024 x 1 13.3 / 14.4 / 7.6, 300 x 2048 x 1
//    20.5 / 23.6 / 8.3, against 1500 x 1024 x 1 38.2 / 14.4 / 22.6).
//  - With more stages few large steps leave SMs idle that the passes through L2 use:
//    20 x 2048 x 10 16.4 / 20.5, 80 x 2048 x 10 22.6 / 20.6, 57 x 1048 x 16 23.6 / 18.5 (217 / 55).
//  - The step form's warps go round the columns of four, six, eight and nine stages with
//    the fewest to spare, and it takes few steps of three long ones: passes / step form
//    300 x 2050 x 4 24.6 / 14.4 (71.8 / 52.4), 330 x 4300 x 4 32.9 / 34.9 (129 / 183),
//    300 x 2500 x 6 28.8 / 22.6 (28.8 / 26.5), 200 x 3600 x 6 28.8 / 30.8, 600 x 2500 x 8
//    56.3 / 59.6 (62.3 / 83.4), 330 x 2500 x 9 61.7 / 74.3 (63.3 / 90.7); 10 x 7000 x 3
//    18.6 / 22.7, 300 x 7000 x 3 69.8 / 28.7.
enum RankForm { kRankPasses, kRankLanes, kRankWarp, kRankColumn, kRankStep };

RankForm rank_form(int64_t T, int64_t R, int64_t S) {
  const int64_t sms = sm_count();
  if (R <= kRankLaneMax) {
    const bool many = T >= sms * 10 ||
                      (R <= 16 ? (S > 16 ? T * 3 >= sms * 10 : S >= 10 ? T >= sms * 5 : S >= 8 && T >= sms * 7)
                               : S > 16 && (R <= 64 ? T * S >= sms * 110 : R <= 96 && T * S >= sms * 160));
    if (!many) return kRankColumn;
    return R >= kRankWarpMin && S <= kRankWarpMaxS ? kRankWarp : kRankLanes;
  }
  const bool step = step_smem(R, S) <= kStepSmemMax;
  if (R <= kColMaxRanks && column_smem(R, S) <= kStepSmemMax) {
    if (step && (S <= 2 ? R > 256 && T < sms * 4 : S <= 4 && R > 1024 && T < sms * 2)) return kRankStep;
    return S > 8 && R > 1250 && T < sms / 2 ? kRankPasses : kRankColumn;
  }
  if (!step || S == 8) return kRankPasses;
  if (S <= 4) return S <= 2 || (S == 4 ? R <= 2500 : R <= 6000 || T >= sms) ? kRankStep : kRankPasses;
  return T >= sms && (S == 6 ? R <= 2500 : S != 9 || R <= 2250) ? kRankStep : kRankPasses;
}

}  // namespace

bool rank_on_chip(int64_t T, int64_t R, int64_t S) { return rank_form(T, R, S) != kRankPasses; }

cudaError_t launch_rank_chip(const int64_t* d, int64_t T, int64_t R, int64_t S, int of_prefix, int64_t t0, int64_t W,
                             int64_t* L, int64_t* dL, int64_t* G, int64_t* Lw, int64_t* Gw, int64_t* spread,
                             uint32_t* status, cudaStream_t stream) {
  ChipParams p{};
  p.d = d;
  p.T = T;
  p.R = static_cast<int>(R);
  p.S = static_cast<int>(S);
  p.of_prefix = of_prefix;
  p.t0 = t0;
  p.W = W;
  p.w_first = t0 / W;
  p.L = L;
  p.dL = dL;
  p.G = G;
  p.Lw = Lw;
  p.Gw = Gw;
  p.spread = spread;
  p.status = status;
  const RankForm form = rank_form(T, R, S);
  if (form == kRankPasses) return cudaErrorInvalidValue;
  if (form == kRankWarp) return launch_rank_warp(p, stream);
  if (form == kRankLanes) return launch_rank_lanes(p, stream);
  if (form == kRankColumn) {
    if (R <= 256) return launch_column<8>(p, stream);
    if (R <= 512) return launch_column<16>(p, stream);
    if (R <= 1024) return launch_column<32>(p, stream);
    return launch_column<64>(p, stream);
  }
  if (S <= 4) return launch_step<4>(p, stream);
  if (S <= 8) return launch_step<8>(p, stream);
  if (S <= 16) return launch_step<16>(p, stream);
  return launch_step<32>(p, stream);
}

}  // namespace sf
