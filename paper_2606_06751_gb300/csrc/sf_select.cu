// sf_select.cu - the per-window kernels of libstagefrontier:
//   * window_median: lower median of every (window, rank, stage) column
//     (the per-rank window baseline of Sec. 4, Eq. 4);
//   * topk: top-k stages by X and (stage, rank) pairs by lead-rank credit E;
//   * gates: App. C label gates, routing and ambiguity sets, fp64 shares/gains;
//   * zero: clears accumulators the library owns the semantics of.
#include <algorithm>
#include <type_traits>

#include <cooperative_groups.h>

#include "sf_device.cuh"
#include "sf_launch.h"
#include "sf_lane_select.cuh"
#include "sf_warp_select.cuh"

namespace sf {

namespace {

__device__ __forceinline__ int64_t imin64(int64_t a, int64_t b) { return a < b ? a : b; }

__global__ void zero_kernel(uint32_t* __restrict__ p, size_t words) {
  for (size_t i = blockIdx.x * size_t(blockDim.x) + threadIdx.x; i < words;
       i += size_t(gridDim.x) * blockDim.x)
    p[i] = 0u;
}

// Clears up to kZeroMax buffers in one launch (a call's accumulators), and
// lets the pass that follows it on the stream start at once (it waits for
// this kernel's completion before its first write).
__global__ void zero_many_kernel(const ZeroList z) {
  griddep_launch_dependents();
  for (int b = 0; b < z.n; ++b) {
    uint32_t* __restrict__ p = static_cast<uint32_t*>(z.ptr[b]);
    for (size_t i = blockIdx.x * size_t(blockDim.x) + threadIdx.x; i < z.words[b];
         i += size_t(gridDim.x) * blockDim.x)
      p[i] = 0u;
  }
}

// ---------------------------------------------------------------------------
// Lower median, one warp per column.  A CTA of 8 warps owns (window w, eight
// consecutive flat columns c = r*S + s).  The window's rows of those columns
// are read coalesced and transposed through shared memory so each warp holds
// its column in registers (NPL values per lane).  Values are mapped to an
// order-preserving unsigned key (so any int64 input is handled exactly) and
// offset by the column minimum; the k-th smallest offset (k = floor((n-1)/2))
// is then found by radix selection, most significant 8-bit digit first: a
// per-warp 256-bin shared-memory histogram of the digit among the values that
// share the digits chosen so far, a warp scan to find the bin holding rank k,
// and the rank re-based into that bin.  A 24-bit spread takes three passes.
constexpr int kMedCols = 8;
constexpr int kMedThreads = kMedCols * 32;
// k-th smallest (0-based) of the lane-strided values get(i) (row lane + 32 i,
// valid while row < n), all below 2^nbits.  hist: this warp's 256 counters.
template <typename U, int NPL, typename Get>
__device__ __forceinline__ U warp_radix_select(Get get, int n, int nbits, uint32_t k, uint32_t* hist,
                                               int lane) {
  U prefix = 0;
  int shift = nbits;
  uint32_t rem = k;
  bool first = true;
  while (shift > 0) {
    const int D = shift < 8 ? shift : 8;
    shift -= D;
    const uint32_t dmask = (1u << D) - 1u;
    const int hs = shift + D;  // bits above the current digit
    reinterpret_cast<uint4*>(hist)[2 * lane] = make_uint4(0, 0, 0, 0);
    reinterpret_cast<uint4*>(hist)[2 * lane + 1] = make_uint4(0, 0, 0, 0);
    __syncwarp();
#pragma unroll
    for (int i = 0; i < NPL; ++i) {
      if (lane + 32 * i < n) {
        const U v = get(i);
        if (first || (v >> hs) == prefix)
          atomicAdd(&hist[static_cast<uint32_t>(v >> shift) & dmask], 1u);
      }
    }
    __syncwarp();
    const uint4 h0 = reinterpret_cast<const uint4*>(hist)[2 * lane];
    const uint4 h1 = reinterpret_cast<const uint4*>(hist)[2 * lane + 1];
    const uint32_t hb[8] = {h0.x, h0.y, h0.z, h0.w, h1.x, h1.y, h1.z, h1.w};
    uint32_t sum = 0;
#pragma unroll
    for (int j = 0; j < 8; ++j) sum += hb[j];
    uint32_t incl = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t up = __shfl_up_sync(kFull, incl, o);
      if (lane >= o) incl += up;
    }
    const uint32_t excl = incl - sum;
    const int owner = __ffs(__ballot_sync(kFull, excl <= rem && rem < incl)) - 1;
    uint32_t digit = 0, below = excl;
    if (lane == owner) {
      uint32_t c = excl;
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        if (rem >= c && rem < c + hb[j]) {
          digit = 8u * lane + j;
          below = c;
        }
        c += hb[j];
      }
    }
    digit = __shfl_sync(kFull, digit, owner);
    below = __shfl_sync(kFull, below, owner);
    rem -= below;
    prefix = (prefix << D) | static_cast<U>(digit);
    first = false;
    __syncwarp();
  }
  return prefix;
}

template <int NPL, bool kVec>
__global__ void __launch_bounds__(kMedThreads)
    median_kernel(const int64_t* __restrict__ d, int64_t T, int64_t RS, int64_t W, int64_t ngroups,
                  int64_t* __restrict__ m) {
  constexpr int LD = 32 * NPL + 1;
  extern __shared__ int64_t colbuf[];  // [kMedCols][LD], then kMedCols x 256 histogram counters
  // kMedCols * LD * 8 bytes is a multiple of 64, so the counters start 16-byte aligned
  uint32_t* hists = reinterpret_cast<uint32_t*>(colbuf + kMedCols * LD);
  const int64_t w = blockIdx.x / ngroups;
  const int64_t c0 = (blockIdx.x % ngroups) * kMedCols;
  const int ncols = static_cast<int>(imin64(kMedCols, RS - c0));
  const int64_t tb = w * W;
  const int n = static_cast<int>(imin64(W, T - tb));
  const int64_t* base = d + tb * RS + c0;
  if (kVec && ncols == kMedCols) {  // 16-byte loads of column pairs (RS even)
    for (int idx = threadIdx.x; idx < n * (kMedCols / 2); idx += kMedThreads) {
      const int row = idx / (kMedCols / 2), pr = idx % (kMedCols / 2);
      const longlong2 v = __ldg(reinterpret_cast<const longlong2*>(base + int64_t(row) * RS) + pr);
      colbuf[(2 * pr) * LD + row] = v.x;
      colbuf[(2 * pr + 1) * LD + row] = v.y;
    }
  } else {
    for (int idx = threadIdx.x; idx < n * kMedCols; idx += kMedThreads) {
      const int row = idx / kMedCols, c = idx % kMedCols;
      colbuf[c * LD + row] = c < ncols ? __ldg(base + int64_t(row) * RS + c) : 0;
    }
  }
  __syncthreads();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (warp >= ncols) return;
  uint32_t* hist = hists + warp * kSelBins;  // 1 KB per warp
  constexpr uint64_t kSign = 1ull << 63;
  uint64_t u[NPL];
  uint64_t lo = ~0ull, hi = 0;
#pragma unroll
  for (int i = 0; i < NPL; ++i) {
    const int row = lane + 32 * i;
    u[i] = row < n ? static_cast<uint64_t>(colbuf[warp * LD + row]) ^ kSign : 0;
    if (row < n) {
      lo = u[i] < lo ? u[i] : lo;
      hi = u[i] > hi ? u[i] : hi;
    }
  }
  lo = warp_min_u64(lo);
  hi = warp_max_u64(hi);
  const uint32_t k = static_cast<uint32_t>((n - 1) / 2);
  const uint64_t range = hi - lo;
  const int nbits = range ? 64 - __clzll(static_cast<long long>(range)) : 0;
  uint64_t ans;
  if (nbits <= 32) {
    uint32_t x[NPL];
#pragma unroll
    for (int i = 0; i < NPL; ++i) x[i] = static_cast<uint32_t>(u[i] - lo);  // padding rows never read
    ans = warp_radix_select<uint32_t, NPL>([&](int i) { return x[i]; }, n, nbits, k, hist, lane);
  } else {
#pragma unroll
    for (int i = 0; i < NPL; ++i) u[i] -= lo;
    ans = warp_radix_select<uint64_t, NPL>([&](int i) { return u[i]; }, n, nbits, k, hist, lane);
  }
  if (lane == 0) m[w * RS + c0 + warp] = static_cast<int64_t>((lo + ans) ^ kSign);
}

// Lower median of one column of n <= 32 NPL rows read from global memory
// (stride RS) on every pass, on 64-bit order-preserving keys: the path of a
// column whose values do not share their high 32 bits.  Kept out of line so
// its registers do not weigh on the 32-bit path.
template <int NPL>
__device__ __noinline__ int64_t median_column_global(const int64_t* __restrict__ dc, int64_t RS, int n, uint32_t* hist,
                                                     int lane) {
  constexpr uint64_t kSign = 1ull << 63;
  auto ukey = [&](int i) { return static_cast<uint64_t>(__ldg(dc + int64_t(lane + 32 * i) * RS)) ^ kSign; };
  uint64_t lo = ~0ull, hi = 0;
#pragma unroll 4
  for (int i = 0; i < NPL; ++i)
    if (lane + 32 * i < n) {
      const uint64_t u = ukey(i);
      lo = u < lo ? u : lo;
      hi = u > hi ? u : hi;
    }
  lo = warp_min_u64(lo);
  hi = warp_max_u64(hi);
  const uint64_t range = hi - lo;
  const int nbits = range ? 64 - __clzll(static_cast<long long>(range)) : 0;
  const uint32_t k = static_cast<uint32_t>((n - 1) / 2);
  const uint64_t key =
      lo + warp_radix_select<uint64_t, NPL>([&](int i) { return ukey(i) - lo; }, n, nbits, k, hist, lane);
  return static_cast<int64_t>(key ^ kSign);
}

// A column of the tile whose values do not share their high words, most often
// for a few outliers alone (one stall of seconds among milliseconds): row 0's
// high word is tried for the median's.  Larger values become the largest of the
// column that share it, smaller ones the smallest, in the tile, which moves the
// median only if it is not among the sharers; returns false, with the tile as it
// was, if it is not.  row0: the column's place in the tile's first row.
__device__ __noinline__ bool clamp_column(unsigned char* row0, uint32_t swizzle_bits, int n, int lane) {
  // rows are 64 bytes apart, their 16-byte chunks permuted by bits 1-2 of the row
  auto at = [&](int r) {
    return reinterpret_cast<uint2*>(row0 + r * 64 + (((swizzle_bits >> 1) ^ ((r >> 1) & 3)) << 4) + ((swizzle_bits & 1) << 3));
  };
  const uint32_t h0 = at(0)->y, k = static_cast<uint32_t>((n - 1) / 2);
  uint32_t same = 0, under = 0, lo = 0xffffffffu, hi = 0;
#pragma unroll 4
  for (int r = lane; r < n; r += 32) {
    const uint2 v = *at(r);
    if (v.y == h0) {
      ++same;
      lo = min(lo, v.x);
      hi = max(hi, v.x);
    } else if (static_cast<int32_t>(v.y) < static_cast<int32_t>(h0)) {
      ++under;
    }
  }
  same = __reduce_add_sync(kFull, same);
  under = __reduce_add_sync(kFull, under);
  if (k < under || k - under >= same) return false;
  lo = __reduce_min_sync(kFull, lo);
  hi = __reduce_max_sync(kFull, hi);
#pragma unroll 4
  for (int r = lane; r < n; r += 32) {
    const uint2 v = *at(r);
    if (v.y != h0) *at(r) = make_uint2(static_cast<int32_t>(v.y) < static_cast<int32_t>(h0) ? lo : hi, h0);
  }
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // before the next tile's copies
  __syncwarp();
  return true;
}

// Persistent form of the median: each CTA walks (window, 8-column) tiles
// with one tile buffer and two mbarriers.  `full` completes when a tile's
// bulk copies have landed; each warp copies its column into registers and
// arrives on `empty`, and once all eight have, one thread issues the copies
// of the CTA's next tile into the same buffer, so the copy runs under the
// selection of the current tile and no CTA-wide barrier aligns the warps.
// The selection touches only registers and the warp's counters.  A column
// whose median is not among the values that share row 0's high 32 bits selects
// on 64-bit values re-read from d (all columns with an outlier past 32 bits did:
// a heavy-tailed 50000 x 1024 x 10, W = 500, 1352 us).  Past 512 rows and without
// kFit, any column whose values do not share them does: there the loop that reads a
// clamped column once more took 4 to 18 % of every other column (3430 x 3128 x 8,
// W = 343, 247 -> 211 us without it; out of line 232).  Every window of a launch
// holds the same n rows.
//
// Resident CTAs hide each tile's copy and selection chain, so the registers are
// held to what the most CTAs allow without spilling the column (512-row columns,
// 1024 x 10: three CTAs 832 us, four 824 us).
constexpr int med_min_ctas(int npl) { return npl >= 32 ? 3 : npl == 16 ? 4 : 5; }

template <int NPL, bool kFit>
__global__ void __launch_bounds__(kMedThreads, med_min_ctas(NPL))
    median_persist_kernel(const __grid_constant__ CUtensorMap map, const int64_t* __restrict__ d, int64_t T,
                          int64_t RS, int64_t W, int64_t w0, int64_t nW, int64_t ngroups, int box_rows, int nbox,
                          int64_t* __restrict__ m, uint32_t* status) {
  extern __shared__ unsigned char smem_raw[];
  unsigned char* tile = align_1024(smem_raw);
  const uint32_t tile_bytes = uint32_t(nbox) * uint32_t(box_rows) * 64u;  // bytes the copies write
  const int tile_rows = max(nbox * box_rows, 32 * NPL);
  uint32_t* hists = reinterpret_cast<uint32_t*>(tile + uint32_t(tile_rows) * 64u);
  uint64_t* full = reinterpret_cast<uint64_t*>(hists + kMedCols * kSelHistWords);
  uint64_t* empty = full + 1;
  volatile int* abort = reinterpret_cast<volatile int*>(full + 2);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  uint32_t* hist = hists + warp * kSelHistWords;
  // Tile numbers, columns of a step and windows of a launch fit 32 bits (the entry
  // point's limits): shorter divisions, fewer registers (512 rows: 824 -> 803 us).
  // With 32 slots that made the compiler spill the column, twice the time.
  using Id = std::conditional_t<(NPL > 16), int64_t, uint32_t>;
  const Id groups = static_cast<Id>(ngroups), ntiles = static_cast<Id>(nW) * groups;
  auto issue = [&](Id id) {  // one thread: the bulk copies of tile `id`
    const Id c0 = (id % groups) * kMedCols;
    const int64_t tb = (w0 + id / groups) * W;
    mbar_arrive_expect_tx(full, tile_bytes);
    for (int b = 0; b < nbox; ++b)
      tma_load_2d(tile + size_t(b) * box_rows * 64, &map, static_cast<int32_t>(c0),
                  static_cast<int32_t>(tb + int64_t(b) * box_rows), full);
  };
  if (threadIdx.x == 0) {
    mbar_init(full, 1);
    mbar_init(empty, kMedCols);
    *abort = 0;
    fence_barrier_init();
  }
  __syncthreads();
  bool issued = blockIdx.x < ntiles;  // (thread 0) the copies of the awaited tile were issued
  if (threadIdx.x == 0 && issued) issue(blockIdx.x);
  const unsigned char* col = tile + lane * 64u + ((((warp >> 1) ^ ((lane >> 1) & 3)) << 4) | ((warp & 1) << 3));
  uint32_t phase = 0;
  for (Id id = blockIdx.x; id < ntiles; id += gridDim.x, phase ^= 1u) {
    const int64_t w = w0 + id / groups;
    const Id c0 = (id % groups) * kMedCols;
    const bool mine = warp < imin64(kMedCols, RS - c0);
    const int n = static_cast<int>(imin64(W, T - w * W));
    // a warp goes on only if all its lanes saw the tile (a wait gives up
    // after its time limit, or at once when another thread has)
    if (!__all_sync(kFull, mbar_wait_bounded(full, phase, abort))) {
      if (threadIdx.x == 0) {
        report(status, SF_ST_TIMEOUT);
        if (issued) mbar_wait_timeout(full, phase);  // let the copies land before the CTA's memory is released
      }
      return;
    }
    // Slot i holds a row of the window iff lane + 32 i < n (with kFit, only
    // the last slot can fail it).  A padding slot repeats a live value; the
    // high words agree iff their AND equals their OR over the column.
    auto live = [&](int i) { return (kFit && i + 1 < NPL) || lane + 32 * i < n; };
    uint32_t xl[NPL];
    uint32_t hand, hor, live_x = 0u;
    for (bool again = NPL <= 16 && kFit && mine;; again = false) {
      hand = 0xffffffffu;
      hor = 0u;
#pragma unroll
      for (int i = 0; i < NPL; ++i) {
        const uint2 v = *reinterpret_cast<const uint2*>(col + i * 2048);  // in the tile even past the window
        if (i == 0) live_x = kFit && NPL >= 2 ? v.x : __shfl_sync(kFull, v.x, 0);  // row 0 is in every window
        const bool okr = live(i);
        xl[i] = okr ? v.x : live_x;
        hand &= okr ? v.y : 0xffffffffu;
        hor |= okr ? v.y : 0u;
      }
      // with kFit, a column whose high words differ is clamped and read once more (not
      // with 32 slots: the call's registers would spill them)
      if (NPL > 16 || !kFit || !again || __reduce_and_sync(kFull, hand) == __reduce_or_sync(kFull, hor) ||
          !clamp_column(tile, static_cast<uint32_t>(warp), n, lane))
        break;
    }
    __syncwarp();
    if (lane == 0) mbar_arrive(empty);  // this warp is done with the buffer
    const Id next = id + gridDim.x;
    if (threadIdx.x == 0 && next < ntiles) {
      issued = mbar_wait_bounded(empty, phase, abort);
      if (issued) issue(next);  // else the abort flag is set and every warp leaves at its next wait
    }
    if (!mine) continue;
    const uint32_t hw = __reduce_and_sync(kFull, hand);
    const uint32_t k = static_cast<uint32_t>((n - 1) / 2);
    if (hw == __reduce_or_sync(kFull, hor)) {
      uint32_t lmin = xl[0], lmax = xl[0];
#pragma unroll
      for (int i = 1; i + 1 < NPL; i += 2) {
        lmin = __vimin3_u32(lmin, xl[i], xl[i + 1]);
        lmax = __vimax3_u32(lmax, xl[i], xl[i + 1]);
      }
      if ((NPL & 1) == 0) {
        lmin = min(lmin, xl[NPL - 1]);
        lmax = max(lmax, xl[NPL - 1]);
      }
      lmin = __reduce_min_sync(kFull, lmin);
      lmax = __reduce_max_sync(kFull, lmax);
      const uint32_t range = lmax - lmin;
      const int nbits = range ? 32 - __clz(static_cast<int>(range)) : 0;
      const uint32_t pad = nbits == 32 ? 0xffffffffu : (1u << nbits) - 1u;  // sorts at or after every live value
#pragma unroll
      for (int i = 0; i < NPL; ++i) xl[i] = live(i) ? xl[i] - lmin : pad;
      const uint32_t ans = warp_select_regs<NPL>(xl, nbits, k, hist, lane);
      if (lane == 0) m[w * RS + c0 + warp] = static_cast<int64_t>((static_cast<uint64_t>(hw) << 32) | (lmin + ans));
    } else {
      // the buffer may already hold the next tile: re-read the column from d
      const int64_t med = median_column_global<NPL>(d + w * W * RS + c0 + warp, RS, n, hist, lane);
      if (lane == 0) m[w * RS + c0 + warp] = med;
    }
  }
}

// Short windows (n <= 128 rows): one lane per column.  A warp takes 32
// consecutive columns of a window, so its loads are whole 256-byte runs of d at
// any alignment, and every lane holds its column in registers (32-bit keys, the
// values' low words) and searches its own median without a word to the others
// (lane_select).  A column whose values do not share their high words is taken
// by the whole warp on 64-bit values.  Against a warp per column, whose histogram
// and searches cost as much for a hundred rows as for a thousand: 100000 x 128 x 6
// in windows of 100 steps 337 -> 188 us, one window of 100 x 8192 x 8 33 -> 22.5 us.
// Bound by the loads a warp can hold beside its keys.
constexpr int kLaneMedThreads = 128;
constexpr int kLaneMedMaxRows = 128;

template <int NMAX>
__global__ void __launch_bounds__(kLaneMedThreads, lane_ctas(NMAX))
    median_lanes_kernel(const int64_t* __restrict__ d, int64_t T, int64_t RS, int64_t W, int64_t tiles,
                        int64_t ntiles, int64_t* __restrict__ m) {
  constexpr int kBatch = lane_batch(NMAX);  // rows loaded together
  __shared__ __align__(16) uint32_t hists[kLaneMedThreads / 32][kSelHistWords];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t nw = int64_t(gridDim.x) * (kLaneMedThreads / 32);
  for (int64_t id = int64_t(blockIdx.x) * (kLaneMedThreads / 32) + warp; id < ntiles; id += nw) {
    const int64_t w = id / tiles, c0 = (id - w * tiles) * 32, tb = w * W;
    const int n = static_cast<int>(imin64(W, T - tb));
    const bool mine = c0 + lane < RS;
    const int64_t* col = d + tb * RS + c0 + (mine ? lane : 0);
    uint32_t x[NMAX];
    uint32_t hand = 0xffffffffu, hor = 0u;
#pragma unroll
    for (int b = 0; b < NMAX; b += kBatch) {
      uint2 v[kBatch];
#pragma unroll
      for (int i = 0; i < kBatch; ++i) v[i] = load_words(col + min(b + i, n - 1) * RS);  // past the window: its last row
#pragma unroll
      for (int i = 0; i < kBatch; ++i) {
        x[b + i] = b + i < n ? v[i].x : 0xffffffffu;  // sorts last
        hand &= v[i].y;
        hor |= v[i].y;
      }
    }
    const uint32_t kth = static_cast<uint32_t>((n - 1) / 2);
    uint32_t lo = 0xffffffffu, hi = 0u;
#pragma unroll
    for (int i = 0; i < NMAX; ++i) {
      lo = min(lo, x[i]);
      hi = max(hi, i < n ? x[i] : 0u);
    }
    const uint32_t ans = lane_select<NMAX>(x, static_cast<uint32_t>(n), kth, lo, hi);
    const bool split = hand != hor;  // this column's high words differ
    if (mine && !split) m[w * RS + c0 + lane] = static_cast<int64_t>((static_cast<uint64_t>(hor) << 32) | ans);
    for (uint32_t todo = __ballot_sync(kFull, mine && split); todo; todo &= todo - 1) {
      const int64_t c = c0 + __ffs(todo) - 1;
      const int64_t med = median_column_global<(NMAX + 31) / 32>(d + tb * RS + c, RS, n, hists[warp], lane);
      if (lane == 0) m[w * RS + c] = med;
    }
  }
}

template <int NMAX>
cudaError_t launch_median_lanes(const int64_t* d, int64_t T, int64_t RS, int64_t W, int64_t* m, cudaStream_t stream) {
  const int64_t tiles = (RS + 31) / 32, ntiles = (T + W - 1) / W * tiles;
  int per_sm = 0;
  const cudaError_t e =
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, median_lanes_kernel<NMAX>, kLaneMedThreads, 0);
  if (e != cudaSuccess) return e;
  const int64_t warps = kLaneMedThreads / 32;
  const int64_t grid = std::min<int64_t>((ntiles + warps - 1) / warps, int64_t(sm_count()) * std::max(per_sm, 1));
  count_launch();
  median_lanes_kernel<NMAX><<<static_cast<unsigned>(grid), kLaneMedThreads, 0, stream>>>(d, T, RS, W, tiles, ntiles, m);
  return cudaGetLastError();
}

// Windows longer than 1024 steps: the same search, re-reading the column
// from global memory (L2) on every bit.
__global__ void __launch_bounds__(kMedThreads)
    median_global_kernel(const int64_t* __restrict__ d, int64_t T, int64_t RS, int64_t W,
                         int64_t ngroups, int64_t* __restrict__ m) {
  const int64_t w = blockIdx.x / ngroups;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t c = (blockIdx.x % ngroups) * kMedCols + warp;
  if (c >= RS) return;
  const int64_t tb = w * W;
  const int64_t n = imin64(W, T - tb);
  const int64_t* col = d + tb * RS + c;
  constexpr uint64_t kSign = 1ull << 63;
  uint64_t lo = ~0ull, hi = 0;
  for (int64_t t = lane; t < n; t += 32) {
    const uint64_t u = static_cast<uint64_t>(__ldg(col + t * RS)) ^ kSign;
    lo = u < lo ? u : lo;
    hi = u > hi ? u : hi;
  }
  lo = warp_min_u64(lo);
  hi = warp_max_u64(hi);
  const uint64_t k = static_cast<uint64_t>((n - 1) / 2);
  const uint64_t range = hi - lo;
  const int nbits = range ? 64 - __clzll(static_cast<long long>(range)) : 0;
  uint64_t ans = 0;
  for (int bit = nbits - 1; bit >= 0; --bit) {
    const uint64_t cand = ans | (1ull << bit);
    uint32_t cnt = 0;
    for (int64_t t = lane; t < n; t += 32)
      cnt += ((static_cast<uint64_t>(__ldg(col + t * RS)) ^ kSign) - lo) < cand ? 1u : 0u;
    cnt = __reduce_add_sync(kFull, cnt);
    if (cnt <= k) ans = cand;
  }
  if (lane == 0) m[w * RS + c] = static_cast<int64_t>((lo + ans) ^ kSign);
}

// ---------------------------------------------------------------------------
// Top-k.  Order: value descending, then index ascending (index = stage for X,
// s*R + r for E); value 0 is not a suspect.
//
// A window's (stage, rank) entries are split over a cluster of one to
// kTopCluster CTAs (about one tile of entries each, eight at most).  Each CTA reads
// its slice once, kTopTile entries at a time with the next tile's loads in flight,
// and appends the positive entries to a list in
// shared memory: lead-rank credit is sparse (at most one rank per step and
// stage), so a slice's list usually ends far below its capacity.  A list that
// could not take another whole tile is first cut to its k best.  The cut runs
// in registers, warp by warp (k rounds of a warp arg-max, no CTA barrier
// between rounds), then over the warps' k best; the cluster's first CTA merges
// the CTAs' k best through distributed shared memory.  What is left is the
// latency of one pass of loads, three cuts and two cluster barriers: k = 5 of
// 20 windows of 8192 x 8 entries takes 14.5 us (33.2 us as k rounds of a block
// arg-max that each re-read the slice), of one window 10.9 us (20.6 us).
constexpr int kTopThreads = 256;
constexpr int kTopWarps = kTopThreads / 32;
constexpr int kTopCluster = 8;
constexpr int kTopMaxK = 32;
constexpr int kTopPerThread = 8;
constexpr int kTopTile = kTopPerThread * kTopThreads;  // entries read together
constexpr int kTopCap = 3584;                          // list entries (43 KB)
constexpr int kTopSlots = kTopCap / kTopThreads;       // list entries a lane takes in a cut
static_assert(kTopCap % kTopThreads == 0 && kTopCap >= kTopTile + kTopMaxK, "a cut list takes a whole tile");

struct TopShared {
  int64_t v[kTopCap];
  int32_t i[kTopCap];
  int64_t wv[kTopWarps * kTopMaxK];  // each warp's k best
  int32_t wi[kTopWarps * kTopMaxK];
  int n;
};

// a ranks ahead of b
__device__ __forceinline__ bool before(int64_t av, int32_t ai, int64_t bv, int32_t bi) {
  return av > bv || (av == bv && ai < bi);
}

// The k best of the entries base + stride q < m, q = 0..N-1, of lists V and I,
// in order, to ov / oi (value 0 past the last positive one).  Whole warp.
template <int N>
__device__ __forceinline__ void warp_top(const int64_t* V, const int32_t* I, int m, int base, int stride, int k,
                                         int64_t* ov, int32_t* oi, int lane) {
  int64_t v[N];
  int32_t id[N];
#pragma unroll
  for (int q = 0; q < N; ++q) {
    const int at = base + stride * q;
    v[q] = at < m ? V[at] : 0;
    id[q] = at < m ? I[at] : INT32_MAX;
  }
  for (int r = 0; r < k; ++r) {
    int64_t bv = 0;  // this lane's best
    int32_t bi = INT32_MAX;
#pragma unroll
    for (int q = 0; q < N; ++q)
      if (before(v[q], id[q], bv, bi)) {
        bv = v[q];
        bi = id[q];
      }
    const int64_t mv = static_cast<int64_t>(warp_max_u64(static_cast<uint64_t>(bv)));
    const int32_t mi = __reduce_min_sync(kFull, bv == mv ? bi : INT32_MAX);
#pragma unroll
    for (int q = 0; q < N; ++q)
      if (id[q] == mi) v[q] = 0, id[q] = INT32_MAX;  // indices are unique: only the pick goes
    if (lane == 0) {
      ov[r] = mv;
      oi[r] = mi;
    }
  }
  __syncwarp();
}

// Cuts the CTA's list of m entries to its k best, in order.  Every thread calls it.
__device__ __forceinline__ void cut_list(TopShared& sh, int m, int k) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  int64_t* wv = sh.wv + warp * k;
  int32_t* wi = sh.wi + warp * k;
  if (m <= 4 * kTopThreads)
    warp_top<4>(sh.v, sh.i, m, threadIdx.x, kTopThreads, k, wv, wi, lane);
  else
    warp_top<kTopSlots>(sh.v, sh.i, m, threadIdx.x, kTopThreads, k, wv, wi, lane);
  __syncthreads();  // the list has been read, the warps' picks are written
  if (warp == 0) {
    warp_top<kTopMaxK * kTopWarps / 32>(sh.wv, sh.wi, kTopWarps * k, lane, 32, k, sh.v, sh.i, lane);
    if (lane == 0) sh.n = k;
  }
  __syncthreads();
}

__global__ void __launch_bounds__(kTopThreads)
    topk_kernel(const int64_t* __restrict__ X, const int64_t* __restrict__ E, int64_t S, int64_t R, int k,
                int32_t* top_stage, int64_t* top_stage_value, int32_t* top_pair, int64_t* top_pair_value) {
  namespace cg = cooperative_groups;
  cg::cluster_group cluster = cg::this_cluster();
  __shared__ TopShared sh;
  const int csize = static_cast<int>(cluster.num_blocks());
  const int part = static_cast<int>(cluster.block_rank());
  const int64_t w = blockIdx.x / csize;
  const int lane = threadIdx.x & 31;
  const bool pairs = E != nullptr && (top_pair != nullptr || top_pair_value != nullptr);  // uniform over the grid
  const int n = static_cast<int>(S * R);  // <= 2^21
  const int chunk = (n + csize - 1) / csize;
  const int lo = min(part * chunk, n), hi = min(lo + chunk, n);
  const int64_t* Ew = E + w * n;
  int64_t next[kTopPerThread];
  auto load_tile = [&](int at) {
#pragma unroll
    for (int q = 0; q < kTopPerThread; ++q) {
      const int j = at + q * kTopThreads + static_cast<int>(threadIdx.x);
      next[q] = j < hi ? __ldg(Ew + j) : 0;
    }
  };
  if (pairs) load_tile(lo);
  if (part == 0 && threadIdx.x < 32 && (top_stage || top_stage_value)) {
    const int64_t v = lane < S ? X[w * S + lane] : 0;
    bool taken = false;
    for (int i = 0; i < k; ++i) {
      const uint64_t c = (!taken && lane < S && v > 0) ? static_cast<uint64_t>(v) : 0ull;
      const uint64_t mx = warp_max_u64(c);
      int who = -1;
      if (mx != 0) who = __ffs(__ballot_sync(kFull, c == mx)) - 1;  // lowest stage among equals
      if (lane == who) taken = true;
      if (lane == 0) {
        if (top_stage) top_stage[w * k + i] = who;
        if (top_stage_value) top_stage_value[w * k + i] = who >= 0 ? static_cast<int64_t>(mx) : 0;
      }
    }
  }
  if (!pairs) return;
  if (threadIdx.x == 0) sh.n = 0;
  __syncthreads();
  for (int at = lo; at < hi; at += kTopTile) {
    if (sh.n + kTopTile > kTopCap) cut_list(sh, sh.n, k);  // the same count in every thread
    int64_t cur[kTopPerThread];
#pragma unroll
    for (int q = 0; q < kTopPerThread; ++q) cur[q] = next[q];
    if (at + kTopTile < hi) load_tile(at + kTopTile);
    __syncthreads();  // every thread has read the count
#pragma unroll
    for (int q = 0; q < kTopPerThread; ++q) {
      const unsigned hit = __ballot_sync(kFull, cur[q] > 0);
      if (hit == 0) continue;
      int base = 0;
      if (lane == 0) base = atomicAdd(&sh.n, __popc(hit));
      base = __shfl_sync(kFull, base, 0) + __popc(hit & ((1u << lane) - 1u));
      if (cur[q] > 0) {
        sh.v[base] = cur[q];
        sh.i[base] = at + q * kTopThreads + static_cast<int>(threadIdx.x);
      }
    }
    __syncthreads();
  }
  cut_list(sh, sh.n, k);  // the list starts with the slice's k best
  cluster.sync();
  if (part == 0 && threadIdx.x < 32) {
    // the candidates of all CTAs into this CTA's spare lists, then one cut
    for (int c = lane; c < csize * k; c += 32) {
      const unsigned from = static_cast<unsigned>(c / k);
      sh.wv[c] = cluster.map_shared_rank(sh.v, from)[c % k];
      sh.wi[c] = cluster.map_shared_rank(sh.i, from)[c % k];
    }
    __syncwarp();
    warp_top<kTopMaxK * kTopCluster / 32>(sh.wv, sh.wi, csize * k, lane, 32, k, sh.v + kTopMaxK, sh.i + kTopMaxK, lane);
    if (lane < k) {
      const int64_t v = sh.v[kTopMaxK + lane];
      const int32_t i = sh.i[kTopMaxK + lane];
      if (top_pair) {
        top_pair[(w * k + lane) * 2 + 0] = v > 0 ? static_cast<int32_t>(i / R) : -1;
        top_pair[(w * k + lane) * 2 + 1] = v > 0 ? static_cast<int32_t>(i % R) : -1;
      }
      if (top_pair_value) top_pair_value[w * k + lane] = v;
    }
  }
  cluster.sync();  // the other CTAs' candidates stay in place until the merge has read them
}

// ---------------------------------------------------------------------------
// Gates (App. C).  One CTA per window: the CTA scans rank roles and splits the
// window's step leaders into 256 segments whose switch counts are joined in
// order by warp shuffles; the first warp then evaluates the gates, lane s for
// stage s, with exact integer comparisons a*den <op> num*b.  A few dependent
// loads and shuffles are all there is to wait for: 4.3-5.0 us for 1 to 100
// windows, where one thread that joined the segments and walked the stages
// took 15-19 us.
constexpr int kGateThreads = 256;
constexpr int kGateWarps = kGateThreads / 32;

__device__ __forceinline__ bool r_gt(__int128 lhs, sf_ratio r, __int128 rhs) {
  return lhs * r.den > static_cast<__int128>(r.num) * rhs;
}
__device__ __forceinline__ bool r_lt(__int128 lhs, sf_ratio r, __int128 rhs) {
  return lhs * r.den < static_cast<__int128>(r.num) * rhs;
}
__device__ __forceinline__ bool r_ge(__int128 lhs, sf_ratio r, __int128 rhs) {
  return lhs * r.den >= static_cast<__int128>(r.num) * rhs;
}

// The confident steps of a range: their count, the leader changes between
// consecutive ones, the first and the last leader.
struct LeadSeg {
  int e = 0, sw = 0, first = -1, last = -1;
  __device__ __forceinline__ void join(const LeadSeg& o) {  // o follows this range
    if (o.e == 0) return;
    sw += o.sw + (e != 0 && last != o.first ? 1 : 0);
    if (e == 0) first = o.first;
    last = o.last;
    e += o.e;
  }
};

// Joins the segments of `n` (a power of two) consecutive lanes into the first one.
__device__ __forceinline__ void join_lanes(LeadSeg& s, int n) {
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    if (o >= n) break;
    LeadSeg up;
    up.e = __shfl_down_sync(kFull, s.e, o);
    up.sw = __shfl_down_sync(kFull, s.sw, o);
    up.first = __shfl_down_sync(kFull, s.first, o);
    up.last = __shfl_down_sync(kFull, s.last, o);
    if ((threadIdx.x & (2 * o - 1)) == 0) s.join(up);
  }
}

__global__ void __launch_bounds__(kGateThreads) gates_kernel(const GateJob g) {
  __shared__ LeadSeg wseg[kGateWarps];
  const int64_t w = blockIdx.x;
  const int S = static_cast<int>(g.S);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const bool valid = lane < S;
  const int64_t tb = w * g.W, te = min(tb + g.W, g.T), n = te - tb;
  int64_t x = 0, y = 0, D = 0;
  if (warp == 0) {
    x = valid ? g.X[w * S + lane] : 0;
    y = valid ? g.Y[w * S + lane] : 0;
    D = g.D[w];
  }
  LeadSeg seg;
  {
    const int j = threadIdx.x;
    const int64_t sb = tb + n * j / kGateThreads, se = tb + n * (j + 1) / kGateThreads;
#pragma unroll 4
    for (int64_t t = sb; t < se; ++t) {
      const uint8_t sl = g.step_lead[t];
      if (sl & SF_STEP_CONFIDENT) {
        const int ld = sl & 31;
        if (seg.e != 0 && ld != seg.last) ++seg.sw;
        if (seg.e == 0) seg.first = ld;
        seg.last = ld;
        ++seg.e;
      }
    }
  }
  int mixed = 0;
  if (g.role) {
    const int32_t r0 = g.role[0];
#pragma unroll 8
    for (int64_t r = 1 + threadIdx.x; r < g.R; r += kGateThreads) mixed |= g.role[r] != r0;
  }
  join_lanes(seg, 32);
  if (lane == 0) wseg[warp] = seg;
  mixed = __syncthreads_or(mixed);
  if (warp != 0) return;
  seg = lane < kGateWarps ? wseg[lane] : LeadSeg();
  join_lanes(seg, kGateWarps);
  const int64_t e = __shfl_sync(kFull, seg.e, 0), sw = __shfl_sync(kFull, seg.sw, 0);
  const sf_label_config& c = g.cfg;
  const bool high_switch = e >= 2 && r_ge(e, c.gamma_elig, n) && r_gt(sw, c.gamma_switch, e - 1);

  bool tel = g.missing != nullptr && g.missing[w] > c.max_missing_ranks;
  if (g.quality) {
    const uint64_t* q = g.quality + w * 6;
    const unsigned __int128 res = (static_cast<unsigned __int128>(q[1]) << 64) | q[0];
    const unsigned __int128 ovl = (static_cast<unsigned __int128>(q[3]) << 64) | q[2];
    const unsigned __int128 ws = (static_cast<unsigned __int128>(q[5]) << 64) | q[4];
    if (res * static_cast<uint64_t>(c.closure_max.den) > ws * static_cast<uint64_t>(c.closure_max.num)) tel = true;
    if (ovl * static_cast<uint64_t>(c.overlap_max.den) > ws * static_cast<uint64_t>(c.overlap_max.num)) tel = true;
  }
  const bool raw = D < c.denom_floor_ns || D == 0;
  if (raw) tel = true;
  uint32_t lab = SF_LABEL_FRONTIER_ACCOUNTING, route = 0, amb = 0;
  if (tel) lab |= SF_LABEL_TELEMETRY_LIMITED;
  if (mixed) lab |= SF_LABEL_ROLE_AWARE_NEEDED;
  if (raw) {
    lab |= SF_LABEL_RAW_ONLY;
  } else {
    // lowest stage with the largest X (Y): order-preserving unsigned keys
    constexpr uint64_t kSign = 1ull << 63;
    const uint64_t kx = static_cast<uint64_t>(x) ^ kSign, ky = static_cast<uint64_t>(y) ^ kSign;
    const uint64_t mx = warp_max_u64(valid ? kx : 0ull), my = warp_max_u64(valid ? ky : 0ull);
    const int s1 = __ffs(__ballot_sync(kFull, valid && kx == mx)) - 1;
    const int64_t x1 = static_cast<int64_t>(mx ^ kSign), y1 = static_cast<int64_t>(my ^ kSign);
    const uint32_t mA = __ballot_sync(kFull, valid && r_lt(x1 - x, c.eta_A, D));
    const uint32_t mG = __ballot_sync(kFull, valid && r_lt(y1 - y, c.eta_G, D));
    amb = mA | mG;
    // leading-share prefix reaching tau_C: a stage is in it when no stage
    // ranks ahead of it or the sum of those that do falls short
    int64_t ahead = 0;
    bool first = true;
    for (int q = 0; q < S; ++q) {
      const int64_t xq = __shfl_sync(kFull, x, q);
      if (xq > x || (xq == x && q < lane)) {
        ahead += xq;
        first = false;
      }
    }
    route = __ballot_sync(kFull, valid && (first || !r_ge(ahead, c.tau_C, D)));
    const bool hiA = r_gt(x1, c.gamma_A, D);
    const bool loG = r_lt(__shfl_sync(kFull, y, s1), c.gamma_G, D);
    const bool W1 = (c.model_fit_mask >> s1) & 1u;
    const bool gain_tie = __popc(mG) >= 2 && r_ge(y1, c.gamma_G, D);
    if (hiA && loG) lab |= W1 ? SF_LABEL_SYNC_WAIT_DEPENDENT : SF_LABEL_CO_CRITICAL;
    if (hiA && !loG) lab |= SF_LABEL_DIRECT_EXPOSURE;
    if (__popc(mA) >= 2 || gain_tie || high_switch) {
      lab |= SF_LABEL_CO_CRITICAL;
      lab &= ~(SF_LABEL_DIRECT_EXPOSURE | SF_LABEL_SYNC_WAIT_DEPENDENT);
    }
    if (tel || mixed) lab &= ~(SF_LABEL_DIRECT_EXPOSURE | SF_LABEL_SYNC_WAIT_DEPENDENT);
  }
  if (valid) {
    if (g.share) g.share[w * S + lane] = raw ? 0.0 : static_cast<double>(x) / static_cast<double>(D);
    if (g.gain) g.gain[w * S + lane] = raw ? 0.0 : static_cast<double>(y) / static_cast<double>(D);
  }
  if (lane == 0) {
    g.labels[w] = lab;
    g.route_mask[w] = route;
    g.amb_mask[w] = amb;
    if (g.n_confident) g.n_confident[w] = static_cast<int32_t>(e);
    if (g.n_switch) g.n_switch[w] = static_cast<int32_t>(sw);
  }
}

template <int NPL>
cudaError_t launch_median_npl(const int64_t* d, int64_t T, int64_t RS, int64_t W, int64_t nW,
                              int64_t ngroups, int64_t* m, cudaStream_t stream) {
  const size_t smem = size_t(kMedCols) * (32 * NPL + 1) * sizeof(int64_t) +
                      size_t(kMedCols) * kSelBins * sizeof(uint32_t);
  const bool vec = (RS % 2) == 0 && (reinterpret_cast<uintptr_t>(d) % 16) == 0;
  auto kern = vec ? median_kernel<NPL, true> : median_kernel<NPL, false>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem));
  if (e != cudaSuccess) return e;
  kern<<<static_cast<unsigned>(nW * ngroups), kMedThreads, smem, stream>>>(d, T, RS, W, ngroups, m);
  return cudaGetLastError();
}

template <int NPL>
cudaError_t launch_median_tma(const CUtensorMap& map, const int64_t* d, int64_t T, int64_t RS, int64_t W,
                              int64_t w0, int64_t nW, int64_t n, int64_t ngroups, int box_rows, int nbox, int64_t* m, uint32_t* status,
                              cudaStream_t stream) {
  const size_t tile_rows = std::max<size_t>(size_t(nbox) * box_rows, 32 * NPL);  // every slot's row is in the tile
  const size_t smem = 1024 + tile_rows * 64 + size_t(kMedCols) * kSelHistWords * 4 + 32;  // + 2 mbarriers, flag
  auto kern = n > 32 * (NPL - 1) ? median_persist_kernel<NPL, true> : median_persist_kernel<NPL, false>;
  cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(smem));
  if (e != cudaSuccess) return e;
  int per_sm = 0;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kMedThreads, smem);
  if (e != cudaSuccess) return e;
  const int64_t grid = std::min<int64_t>(nW * ngroups, int64_t(sm_count()) * std::max(per_sm, 1));
  count_launch();
  kern<<<static_cast<unsigned>(grid), kMedThreads, smem, stream>>>(map, d, T, RS, W, w0, nW, ngroups, box_rows,
                                                                   nbox, m, status);
  return cudaGetLastError();
}

// Windows [w0, w0 + nW) that each hold n rows: the tensor map's box covers a
// window in up to four 256-row copies; NPL slots per lane hold n rows.
cudaError_t launch_median_windows(const int64_t* d, int64_t T, int64_t RS, int64_t W, int64_t w0, int64_t nW,
                                  int64_t n, int64_t ngroups, int64_t* m, uint32_t* status, cudaStream_t stream,
                                  bool& done) {
  done = false;
  const int nbox = static_cast<int>((n + 255) / 256);
  const int box_rows = static_cast<int>(((n + nbox - 1) / nbox + 15) / 16 * 16);  // 1024-byte boxes
  CUtensorMap map;
  const cuuint64_t gdim[2] = {static_cast<cuuint64_t>(RS), static_cast<cuuint64_t>(T)};
  const cuuint64_t gstride[1] = {static_cast<cuuint64_t>(RS) * 8};
  const cuuint32_t box[2] = {static_cast<cuuint32_t>(kMedCols), static_cast<cuuint32_t>(box_rows)};
  const cuuint32_t estride[2] = {1, 1};
  if (encode_fn()(&map, CU_TENSOR_MAP_DATA_TYPE_INT64, 2, const_cast<int64_t*>(d), gdim, gstride, box, estride,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
    return cudaSuccess;
  done = true;
  if (n <= 32) return launch_median_tma<1>(map, d, T, RS, W, w0, nW, n, ngroups, box_rows, nbox, m, status, stream);
  if (n <= 64) return launch_median_tma<2>(map, d, T, RS, W, w0, nW, n, ngroups, box_rows, nbox, m, status, stream);
  if (n <= 128) return launch_median_tma<4>(map, d, T, RS, W, w0, nW, n, ngroups, box_rows, nbox, m, status, stream);
  if (n <= 256) return launch_median_tma<8>(map, d, T, RS, W, w0, nW, n, ngroups, box_rows, nbox, m, status, stream);
  if (n <= 512) return launch_median_tma<16>(map, d, T, RS, W, w0, nW, n, ngroups, box_rows, nbox, m, status, stream);
  return launch_median_tma<32>(map, d, T, RS, W, w0, nW, n, ngroups, box_rows, nbox, m, status, stream);
}

// Self-test of the bounded wait: every thread waits on an mbarrier phase
// that nothing completes (count 2, one arrival), so the wait must give up
// after limit_ns, record SF_ST_TIMEOUT and let the kernel finish.
__global__ void wait_selftest_kernel(uint64_t limit_ns, uint32_t* status) {
  __shared__ uint64_t bar;
  __shared__ int abort;
  if (threadIdx.x == 0) {
    mbar_init(&bar, 2);
    abort = 0;
    fence_barrier_init();
  }
  __syncthreads();
  if (threadIdx.x == 0) mbar_arrive(&bar);  // one of the two arrivals the phase needs
  const bool ok = mbar_wait_bounded(&bar, 0, &abort, limit_ns);
  if (threadIdx.x == 0) report(status, ok ? 0u : SF_ST_TIMEOUT);
}

}  // namespace

cudaError_t launch_wait_selftest(uint64_t limit_ns, uint32_t* status, cudaStream_t stream) {
  count_launch();
  wait_selftest_kernel<<<1, 64, 0, stream>>>(limit_ns, status);
  return cudaGetLastError();
}

cudaError_t launch_zero(void* p, size_t bytes, cudaStream_t stream) {
  if (bytes == 0) return cudaSuccess;
  const size_t words = bytes / 4;
  const int grid = static_cast<int>(std::min<size_t>((words + 255) / 256, size_t(sm_count()) * 8));
  count_launch();
  zero_kernel<<<grid, 256, 0, stream>>>(static_cast<uint32_t*>(p), words);
  return cudaGetLastError();
}

cudaError_t launch_zero_many(const ZeroList& z, cudaStream_t stream, bool* launched) {
  size_t words = 0;
  for (int b = 0; b < z.n; ++b) words = std::max(words, z.words[b]);
  if (launched) *launched = false;
  if (words == 0) return cudaSuccess;
  if (launched) *launched = true;
  const int grid = static_cast<int>(std::min<size_t>((words + 255) / 256, size_t(sm_count()) * 8));
  count_launch();
  zero_many_kernel<<<grid, 256, 0, stream>>>(z);
  return cudaGetLastError();
}

// Whether windows of n rows take a lane per column.  Fewer tiles than four warps per SM:
// a warp per column spreads further (48 columns by 10 windows 4.3 against 12.3 us).
// Otherwise by estimates of both times: the lanes pay for 32 columns where a step has
// fewer, a warp per column for eight (us, warps / lanes: 10000 windows of 100 rows, 8
// columns 39 / 66, 16 76 / 77, 32 146 / 82, 40 181 / 161; of 20 rows, 8 columns 33 / 19;
// 620 windows of 128 rows, 24 columns 10.3 / 13.9; 46 windows of 100 rows, 576 columns, and
// one of 15 20.0 / 14.1).
bool use_median_lanes(int64_t T, int64_t W, int64_t RS, bool bulk) {
  const int64_t n = std::min(W, T), nW = (T + W - 1) / W;
  const int64_t tiles = nW * ((RS + 31) / 32), groups = nW * ((RS + kMedCols - 1) / kMedCols);
  if (n > kLaneMedMaxRows || tiles < int64_t(sm_count()) * 4) return false;
  const double last = T % W && nW > 1 ? 5.0 : 0.0;  // a short last window is a launch of its own there
  return !bulk || 0.07 * n + tiles * 0.000075 * n < last + groups * 0.00365;
}

cudaError_t launch_window_median(const int64_t* d, int64_t T, int64_t R, int64_t S, int64_t W,
                                 int64_t* m, uint32_t* status, cudaStream_t stream) {
  const int64_t RS = R * S;
  const int64_t nW = (T + W - 1) / W;
  const int64_t ngroups = (RS + kMedCols - 1) / kMedCols;
  const int64_t n = std::min(W, T);
  // Bulk-copy path: rows of d are 16-byte multiples (RS even), d is 16-byte
  // aligned, windows fit the register path, the driver encoder is available.
  // A launch's windows share one row count (the slot tests depend on it), so
  // a short last window gets its own launch.
  const bool bulk = RS % 2 == 0 && reinterpret_cast<uintptr_t>(d) % 16 == 0 && n <= 1024 && T < (int64_t(1) << 31) &&
                    encode_fn() != nullptr;
  if (use_median_lanes(T, W, RS, bulk)) {
    if (n <= 32) return launch_median_lanes<32>(d, T, RS, W, m, stream);
    if (n <= 64) return launch_median_lanes<64>(d, T, RS, W, m, stream);
    if (n <= 104) return launch_median_lanes<104>(d, T, RS, W, m, stream);
    return launch_median_lanes<128>(d, T, RS, W, m, stream);
  }
  if (bulk) {
    const int64_t n_last = T - (nW - 1) * W;
    const int64_t nW_first = n_last == n ? nW : nW - 1;
    bool done = false;
    cudaError_t e = launch_median_windows(d, T, RS, W, 0, nW_first, n, ngroups, m, status, stream, done);
    if (e != cudaSuccess) return e;
    if (done && nW_first == nW) return cudaSuccess;
    if (done) {
      e = launch_median_windows(d, T, RS, W, nW - 1, 1, n_last, ngroups, m, status, stream, done);
      if (e != cudaSuccess || done) return e;
    }
    // no tensor map: every window goes the plain-load way below
  }
  count_launch();
  if (n <= 32) return launch_median_npl<1>(d, T, RS, W, nW, ngroups, m, stream);
  if (n <= 64) return launch_median_npl<2>(d, T, RS, W, nW, ngroups, m, stream);
  if (n <= 128) return launch_median_npl<4>(d, T, RS, W, nW, ngroups, m, stream);
  if (n <= 256) return launch_median_npl<8>(d, T, RS, W, nW, ngroups, m, stream);
  if (n <= 512) return launch_median_npl<16>(d, T, RS, W, nW, ngroups, m, stream);
  if (n <= 1024) return launch_median_npl<32>(d, T, RS, W, nW, ngroups, m, stream);
  median_global_kernel<<<static_cast<unsigned>(nW * ngroups), kMedThreads, 0, stream>>>(d, T, RS, W, ngroups, m);
  return cudaGetLastError();
}

cudaError_t launch_topk(const int64_t* X, const int64_t* E, int64_t nW, int64_t S, int64_t R, int32_t k,
                        int32_t* top_stage, int64_t* top_stage_value, int32_t* top_pair,
                        int64_t* top_pair_value, cudaStream_t stream) {
  // one tile of entries per CTA, at most kTopCluster CTAs: more CTAs than that
  // have nothing to read, and pay for their cut and the cluster's barriers
  // (100 windows of 128 x 8 entries, k = 2: 15.4 us with clusters of eight, 6.4 us
  // with one CTA each)
  const int64_t n = E && (top_pair || top_pair_value) ? S * R : 1;
  unsigned csize = 1;
  while (csize < kTopCluster && int64_t(csize) * kTopTile < n) csize *= 2;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = csize;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(static_cast<unsigned>(nW * csize));
  cfg.blockDim = dim3(kTopThreads);
  cfg.stream = stream;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  count_launch();
  return cudaLaunchKernelEx(&cfg, topk_kernel, X, E, S, R, static_cast<int>(k), top_stage, top_stage_value, top_pair,
                            top_pair_value);
}

cudaError_t launch_gates(const GateJob& job, cudaStream_t stream) {
  count_launch();
  gates_kernel<<<static_cast<unsigned>(job.nW), kGateThreads, 0, stream>>>(job);
  return cudaGetLastError();
}

}  // namespace sf
