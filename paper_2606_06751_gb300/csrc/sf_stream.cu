// sf_stream.cu - the streaming passes over the telemetry tensor d[T][R][S]:
//
//   * frontier pass (Sec. 3 Eq. 1-2): rank-local prefixes in registers, the
//     max-prefix frontier with its lowest attaining rank per boundary, the
//     increments a[t,s], and the fused window aggregation (X, D, E, C, leading
//     stage);
//   * evidence pass (Sec. 4 Eq. 4): the same frontier plus, for every stage s,
//     the makespan after replacing s by the clipped per-rank window median,
//     per-step leader confidence and the telemetry-quality sums (App. A);
//   * routing-baseline pass (Sec. 3 Props 1-2, Sec. 6): per-stage maxima and
//     sums, the slowest rank and rank 0 per window.
//
// Tiled path (sf_tiled.cuh: up to 16 stages, any rank count): tiles of d arrive
// through TMA in a shared-memory ring.  Small steps are handled by one warp per
// tile of whole steps, each warp owning two ring stages; larger steps by one
// warp group per step, spread over one or more tiles, with up to four groups
// taking steps in turn (each group owning its ring stages).  The frontier over
// steps of up to 6 KB takes 2-8 steps per warp instruction (lanes_kernel: groups
// of lanes, one step each).  A few hundred steps over many ranks split each
// step's ranks over a thread-block cluster (split_frontier_kernel).
//
// Generic path (17 to 32 stages; medians that are only 8-byte aligned; few small
// steps that are not whole 128-byte rows; tensors that no tensor map describes): a
// CTA per step, plain global loads or, past 16 stages, a ring of bulk copies.  A lane
// per (step, stage) takes many small steps (sf_step_lanes.cu).  All paths share the per-step
// epilogues.  A pass that follows the clear of its own outputs starts as that
// clear's programmatic dependent and writes only after griddep_wait().
#include <algorithm>
#include <array>
#include <numeric>
#include <type_traits>

#include <cooperative_groups.h>

#include "sf_stream.cuh"

namespace sf {

namespace {

template <int S>
__device__ __forceinline__ void load_global_row(const int64_t* src, int64_t (&v)[S]) {
  if constexpr (S % 2 == 0) {
#pragma unroll
    for (int j = 0; j < S / 2; ++j) {
      const longlong2 x = __ldg(reinterpret_cast<const longlong2*>(src) + j);
      v[2 * j] = x.x;
      v[2 * j + 1] = x.y;
    }
  } else {
#pragma unroll
    for (int j = 0; j < S; ++j) v[j] = __ldg(src + j);
  }
}

// --------------------------------------------------------------------------
// Few steps over many ranks (up to a few hundred steps of large jobs, the
// per-window use of Sec. 3): each step's ranks are split over a thread-block
// cluster of `csize` CTAs, all of them resident at once, so every SM streams and
// no SM owns a whole step more than the others.  CTA j of the cluster reads ranks
// [j R / csize, (j+1) R / csize) with 16-byte loads (8-byte ones for odd stage
// counts; U rows in flight per thread), reduces its packed per-stage keys
// (F << 16 | 65535 - r) to shared memory, and the cluster's first CTA takes
// the maximum over the cluster's keys through distributed shared memory
// (ranks are disjoint, so the largest key still carries the lowest attaining
// rank) and runs the step's epilogue.  No global scratch.
//
// Two rows in flight per thread hold half the registers of four, so that more CTAs
// are resident and steps split further.  That pays where the fullest SM then holds
// fewer ranks and a step has six stages or more, or twelve at the same number: frontier,
// us, four rows / two: 200 x 8192 x 8 22.6 / 18.5, 100 x 8192 x 8 14.4 / 12.3,
// 140 x 5504 x 12 13.9 / 12.3; 140 x 8192 x 8 14.4 / 16.2, 75 x 11818 x 16 30.9 / 37.6;
// 54 x 10000 x 4 7.3 / 8.3, 54 x 14356 x 2 with window sums 8.2 / 12.3.  (Ten stages
// gain with as many CTAs too, 140 x 3000 x 10 10.3 / 8.7.)  Where four rows split a step
// as well and leave a CTA 5000 ranks or more, they are as fast or faster
// (64 x 65536 x 8 44.8 / 47.4, 140 x 16384 x 8 27.3 / 28.4, 23 x 34248 x 16 37.7 / 45.2).
constexpr int kSplitThreads = 256;
constexpr int64_t kSplitLongShare = 5000;  // ranks of a CTA from which four rows are in flight
constexpr int kSplitMaxCluster = 16;  // above 8: a non-portable cluster size, allowed per kernel

template <int S, int U>
__global__ void __launch_bounds__(kSplitThreads) split_frontier_kernel(const int64_t* __restrict__ d, const Params p) {
  namespace cg = cooperative_groups;
  cg::cluster_group cl = cg::this_cluster();
  __shared__ uint64_t wkey[kSplitThreads / 32][S];
  __shared__ uint64_t ckey[S];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int csize = static_cast<int>(cl.num_blocks());
  const int j = static_cast<int>(cl.block_rank());
  const int64_t t = blockIdx.x / csize;
  const int64_t R = p.R;
  const int64_t r0 = R * j / csize, r1 = R * (j + 1) / csize;
  const int64_t* dt = d + t * R * S;
  FrontierRows<S> fr;
  fr.init();
  uint32_t dor = 0, tor = 0;
  for (int64_t r = r0 + threadIdx.x; r < r1; r += int64_t(kSplitThreads) * U) {
    int64_t v[U][S];
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (r + int64_t(kSplitThreads) * u < r1) load_global_row<S>(dt + (r + int64_t(kSplitThreads) * u) * S, v[u]);
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (r + int64_t(kSplitThreads) * u < r1) fr.row(v[u], static_cast<int32_t>(r + kSplitThreads * u), dor, tor);
  }
#pragma unroll
  for (int s = 0; s < S; ++s) {
    const uint64_t km = warp_max_u64(fr.key(s));
    if (lane == 0) wkey[warp][s] = km;
  }
  __syncthreads();
  if (threadIdx.x < S) {
    uint64_t k = 0;
    for (int w = 0; w < kSplitThreads / 32; ++w) k = wkey[w][threadIdx.x] > k ? wkey[w][threadIdx.x] : k;
    ckey[threadIdx.x] = k;
  }
  cl.sync();  // every CTA's keys are visible to the cluster
  if (j == 0 && warp == 0) {
    griddep_wait();  // outputs cleared by the launch before this one (when it is its dependent)
    uint64_t key = 0;
    if (lane < S)
      for (int q = 0; q < csize; ++q) {
        const uint64_t k = *cl.map_shared_rank(&ckey[lane], static_cast<unsigned>(q));
        key = k > key ? k : key;
      }
    WinAcc acc;
    finalize_frontier(p, S, t, key, lane, acc);
    if (p.X) flush_window(p, S, acc, lane);
  }
  cl.sync();  // the other CTAs' shared memory stays alive until the first CTA has read it
  const uint32_t bits = range_bits(__reduce_or_sync(kFull, dor), __reduce_or_sync(kFull, tor));
  if (lane == 0) report(p.status, bits);
}

template <int S, int U>
cudaError_t launch_split(const int64_t* d, const Params& p, int csize, cudaStream_t stream, bool pdl) {
  static bool ready = false;  // attribute set once per process (same on every GB300)
  if (!ready) {
    const cudaError_t e = cudaFuncSetAttribute(split_frontier_kernel<S, U>,
                                               cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
    ready = true;
  }
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = static_cast<unsigned>(csize);
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;  // see launch_ex
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.gridDim = dim3(static_cast<unsigned>(p.T * csize));
  cfg.blockDim = dim3(kSplitThreads);
  cfg.stream = stream;
  cfg.attrs = attr;
  cfg.numAttrs = pdl ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, split_frontier_kernel<S, U>, d, p);
}

// Cluster size for T steps over R ranks: the largest size (<= 16, at least
// 512 ranks per CTA) at which all T clusters are resident at once, 0 if none.  A
// cluster is placed within one GPC, so sizes that do not divide a GPC's CTA
// slots evenly fit fewer clusters than the SM count suggests, and a second
// wave of clusters costs more than the parallelism gained (100 steps x 8192
// ranks: 1, 3, 6 and 12 CTAs per step ran at 20.6, 21.9, 25.0 and 28.3 us).
// The resident counts come from the occupancy calculator, once per process.
template <int S, int U>
int split_cluster_size(int64_t T, int64_t R) {
  static const std::array<int, kSplitMaxCluster + 1> fit = [] {
    std::array<int, kSplitMaxCluster + 1> f{};
    if (cudaFuncSetAttribute(split_frontier_kernel<S, U>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) !=
        cudaSuccess) {
      cudaGetLastError();
      return f;
    }
    for (int c = 1; c <= kSplitMaxCluster; ++c) {
      cudaLaunchConfig_t cfg = {};
      cudaLaunchAttribute attr[1];
      attr[0].id = cudaLaunchAttributeClusterDimension;
      attr[0].val.clusterDim.x = static_cast<unsigned>(c);
      attr[0].val.clusterDim.y = 1;
      attr[0].val.clusterDim.z = 1;
      cfg.gridDim = dim3(static_cast<unsigned>(c));
      cfg.blockDim = dim3(kSplitThreads);
      cfg.attrs = attr;
      cfg.numAttrs = 1;
      int n = 0;
      if (cudaOccupancyMaxActiveClusters(&n, split_frontier_kernel<S, U>, &cfg) != cudaSuccess) {
        cudaGetLastError();
        n = 0;
      }
      f[c] = n;
    }
    return f;
  }();
  int best = fit[1] >= T ? 1 : 0;
  for (int c = 2; c <= kSplitMaxCluster; ++c)
    if (R / c >= 512 && fit[c] >= T) best = c;
  return best;
}

template <int U>
int split_cluster(int S, int64_t T, int64_t R) {
  switch (S) {
    case 2: return split_cluster_size<2, U>(T, R);
    case 3: return split_cluster_size<3, U>(T, R);
    case 4: return split_cluster_size<4, U>(T, R);
    case 5: return split_cluster_size<5, U>(T, R);
    case 6: return split_cluster_size<6, U>(T, R);
    case 7: return split_cluster_size<7, U>(T, R);
    case 8: return split_cluster_size<8, U>(T, R);
    case 9: return split_cluster_size<9, U>(T, R);
    case 10: return split_cluster_size<10, U>(T, R);
    case 11: return split_cluster_size<11, U>(T, R);
    case 12: return split_cluster_size<12, U>(T, R);
    case 14: return split_cluster_size<14, U>(T, R);
    case 16: return split_cluster_size<16, U>(T, R);
    default: return 0;
  }
}

template <int U>
cudaError_t dispatch_split(int S, const int64_t* d, const Params& p, int csize, cudaStream_t stream, bool pdl) {
  switch (S) {
    case 2: return launch_split<2, U>(d, p, csize, stream, pdl);
    case 3: return launch_split<3, U>(d, p, csize, stream, pdl);
    case 4: return launch_split<4, U>(d, p, csize, stream, pdl);
    case 5: return launch_split<5, U>(d, p, csize, stream, pdl);
    case 6: return launch_split<6, U>(d, p, csize, stream, pdl);
    case 7: return launch_split<7, U>(d, p, csize, stream, pdl);
    case 8: return launch_split<8, U>(d, p, csize, stream, pdl);
    case 9: return launch_split<9, U>(d, p, csize, stream, pdl);
    case 10: return launch_split<10, U>(d, p, csize, stream, pdl);
    case 11: return launch_split<11, U>(d, p, csize, stream, pdl);
    case 12: return launch_split<12, U>(d, p, csize, stream, pdl);
    case 14: return launch_split<14, U>(d, p, csize, stream, pdl);
    case 16: return launch_split<16, U>(d, p, csize, stream, pdl);
    default: return cudaErrorInvalidValue;
  }
}

// Whether a pass is split, and how: cluster size and rows in flight.  Any T that
// is resident at once up to 12 stages (us, tiles / split: 160 x 8192 x 8 26.7 / 18.4,
// 360 x 5965 x 8 36.8 / 28.9, 200 x 12345 x 6 36.8 / 22.8, 400 x 4001 x 4 16.6 / 10.4,
// 300 x 5000 x 12 31.9 / 28.0, 200 x 5001 x 5 16.6 / 10.3, 360 x 5965 x 7 32.8 / 26.7,
// 100 x 8001 x 7 18.5 / 10.4); with more, whose rows of 128 bytes a lane the loads
// serve badly, only fewer steps than SMs (300 x 4000 x 16 33.0 / 39.0,
// 160 x 16384 x 16 82 / 134).
struct Split {
  int csize = 0;
  int rows = 0;
};

Split plan_split(const StreamJob& j, int sms) {
  Split q;
  if (j.gain || j.base || j.R < 1024 || j.S > 16 || (j.S > 12 && j.T >= sms) || j.T > int64_t(sms) * 8) return q;
  if (j.S % 2 == 0 && reinterpret_cast<uintptr_t>(j.d) % 16 != 0) return q;
  const int S = static_cast<int>(j.S);
  q.rows = 4;
  q.csize = split_cluster<4>(S, j.T, j.R);
  if (q.csize > 1 && j.R / q.csize >= kSplitLongShare) return q;
  const int more = split_cluster<2>(S, j.T, j.R);
  auto busiest = [&](int c) { return double((j.T * c + sms - 1) / sms) * j.R / c; };  // ranks of the fullest SM
  if (q.csize == 0 || (S == 10 && more == q.csize) ||
      (more > q.csize && (S >= 12 ? busiest(more) <= busiest(q.csize) : S >= 6 && busiest(more) <= 0.87 * busiest(q.csize)))) {
    q.rows = 2;
    q.csize = more;
  }
  return q;
}

// --------------------------------------------------------------------------
// Untiled bulk copy global -> shared (both 16-byte aligned, a multiple of 16
// bytes), completion counted in bytes on `bar`.
__device__ __forceinline__ void bulk_load(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                   smem_u32(dst)),
               "l"(reinterpret_cast<uint64_t>(src)), "r"(bytes), "r"(smem_u32(bar))
               : "memory");
}

// Orders this CTA's earlier shared-memory accesses (generic proxy) before
// later bulk copies into shared memory (async proxy).
__device__ __forceinline__ void fence_proxy_async_smem() {
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

// Generic path: any S <= 32, any R; one CTA of 256 threads per step range.
// The per-stage state is sized by the bound SMAX >= S (4, 8, 16 or 32) and
// every stage loop is unrolled to SMAX with an `s < S` guard, so the state
// stays in registers.
constexpr int kGenThreads = 256;

// RING: the CTA's steps are one contiguous byte range of d, streamed with
// bulk copies in kGenRingStages chunks of p.stage_bytes (a power of two) into
// a shared-memory ring; rows are read from the ring at their offset in that
// range (a row may straddle chunks), and only a row past the range's last
// 16-byte boundary is read from global memory.  Thread 0 refills the chunks
// the finished step no longer needs right after the step's closing barrier,
// so no stage is overwritten while a thread still reads it.  A step must fit
// in kGenRingStages - 1 chunks (checked by the host).
constexpr uint32_t kGenRingStages = 8;

template <int SMAX, int MODE, bool VEC, bool RING>
__global__ void __launch_bounds__(kGenThreads)
    stream_generic_kernel(const int64_t* __restrict__ d, const Params p) {
  constexpr bool GAIN = MODE == 1;
  constexpr bool BASE = MODE == 2;
  constexpr uint32_t NST = kGenRingStages;
  __shared__ uint64_t red[kGenThreads / 32][66];
  __shared__ uint64_t full[RING ? NST : 1];
  __shared__ int abort_word;
  extern __shared__ __align__(128) unsigned char ring[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int S = static_cast<int>(p.S);
  const int64_t R = p.R;
  const int64_t G = gridDim.x, b = blockIdx.x;
  const int64_t t_begin = p.T * b / G, t_end = p.T * (b + 1) / G;
  uint32_t dor = 0, tor = 0;
  WinAcc acc;
  QualAcc qa;
  WinTrack qt;  // window of the step a warp is on (evidence pass)
  BaseAcc bacc;
  // ring geometry (RING only): bytes [A0, B0) of d, chunk c in stage c % NST
  const int64_t RS8 = R * S * 8;
  const uint32_t CB = static_cast<uint32_t>(p.stage_bytes);
  const uint32_t cshift = RING ? static_cast<uint32_t>(__ffs(static_cast<int>(CB)) - 1) : 0u;
  const uint32_t RBmask = NST * CB - 1;
  const int64_t A0 = (t_begin * RS8) & ~int64_t(15), B0 = (t_end * RS8) & ~int64_t(15);
  const int64_t nchunks = RING && B0 > A0 ? (B0 - A0 + CB - 1) >> cshift : 0;
  const unsigned char* dbytes = reinterpret_cast<const unsigned char*>(d);
  volatile int* abort = &abort_word;
  int64_t issued = 0, released = 0;  // thread 0: chunks issued; chunks no step needs any more
  auto issue = [&](int64_t c) {
    const uint32_t st = static_cast<uint32_t>(c) & (NST - 1);
    const int64_t off = A0 + (c << cshift);
    const uint32_t bytes = static_cast<uint32_t>(min(int64_t(CB), B0 - off));
    mbar_arrive_expect_tx(&full[st], bytes);
    bulk_load(ring + size_t(st) * CB, dbytes + off, bytes, &full[st]);
  };
  if constexpr (RING) {
    if (threadIdx.x == 0) {
      for (uint32_t i = 0; i < NST; ++i) mbar_init(&full[i], 1);
      *abort = 0;
      fence_barrier_init();
    }
    __syncthreads();
    if (threadIdx.x == 0)
      while (issued < nchunks && issued < int64_t(NST)) issue(issued++);
  }
  griddep_wait();  // outputs cleared by the launch before this one (when it is its dependent)
  for (int64_t t = t_begin; t < t_end; ++t) {
    const int64_t w = GAIN ? qt.at(t, 0, p.W, 0) : 0;
    if (GAIN && p.quality) qual_window(p, qa, w, lane);
    const int64_t s0 = t * RS8;  // the step's first byte
    bool have = true;
    if constexpr (RING) {
      const int64_t s1 = min(s0 + RS8, B0);
      if (s1 > s0)
        for (int64_t c = (s0 - A0) >> cshift; c <= (s1 - 1 - A0) >> cshift; ++c)
          have &= mbar_wait_bounded(&full[static_cast<uint32_t>(c) & (NST - 1)],
                                    static_cast<uint32_t>(c >> ceil_log2(NST)) & 1u, abort);
    }
    // one rank row's durations: from the ring when the whole row lies below
    // B0 (ring offsets wrap), else from global memory
    auto in_ring = [&](int64_t r) { return RING && s0 + (r + 1) * S * 8 <= B0; };
    auto ring_off = [&](int64_t r) { return static_cast<uint32_t>(s0 + r * S * 8 - A0) & RBmask; };
    int64_t b0[SMAX], b1[SMAX];
    int32_t br[SMAX];
    uint64_t slow = 0;
#pragma unroll
    for (int s = 0; s < SMAX; ++s) {
      b0[s] = BASE ? 0 : -1;
      b1[s] = 0;
      br[s] = 0;
    }
    if constexpr (!VEC) {
      // one rank row at a time per thread, in increasing rank order (a strict
      // '>' keeps the lowest rank), each duration loaded where it is used
      for (int64_t r = threadIdx.x; r < R; r += kGenThreads) {
        const int64_t* row = d + (t * R + r) * S;
        const bool rr = in_ring(r);
        const uint32_t ro = RING ? ring_off(r) : 0u;
        auto val = [&](int s) -> int64_t {
          if (RING && rr) return *reinterpret_cast<const int64_t*>(ring + ((ro + 8u * s) & RBmask));
          return __ldg(row + s);
        };
        int64_t P = 0, other = 0;
#pragma unroll
        for (int s = 0; s < SMAX; ++s) {
          if (s >= S) break;
          const int64_t v = have ? val(s) : 0;
          dor |= hi32(v);
          P += v;
          if (s == p.other_stage) other = v;
          if (BASE) {
            b0[s] = v > b0[s] ? v : b0[s];
            b1[s] += v;
          } else if (P > b0[s]) {
            b0[s] = P;
            br[s] = static_cast<int32_t>(r);
          }
        }
        tor |= hi32(P);
        if (BASE) {
          const uint64_t k = (static_cast<uint64_t>(P) << 16) | static_cast<uint64_t>(65535 - r);
          slow = k > slow ? k : slow;
        }
        if (GAIN) {
          const int64_t* mr = p.m + (w * R + r) * S;
#pragma unroll
          for (int s = 0; s < SMAX; ++s) {
            if (s >= S) break;
            int64_t cut = (have ? val(s) : 0) - __ldg(mr + s);
            cut = cut > 0 ? cut : 0;
            b1[s] = (P - cut) > b1[s] ? (P - cut) : b1[s];
          }
          if (p.quality) qual_row(p, qa, t, r, P, other, dor);
        }
      }
    } else {
      // even S (frontier and baseline passes): rows start 16-byte aligned and
      // are loaded whole with 16-byte loads, one row in flight per thread
      static_assert(!GAIN, "the evidence pass loads durations where it uses them");
      for (int64_t r = threadIdx.x; r < R; r += kGenThreads) {
        const int64_t* row = d + (t * R + r) * S;
        const bool rr = in_ring(r);
        const uint32_t ro = RING ? ring_off(r) : 0u;
        int64_t v[SMAX];
#pragma unroll
        for (int s = 0; s < SMAX; s += 2) {
          if (s >= S) break;
          longlong2 x = make_longlong2(0, 0);
          if (RING && rr) {
            if (have) x = *reinterpret_cast<const longlong2*>(ring + ((ro + 8u * s) & RBmask));
          } else {
            x = __ldg(reinterpret_cast<const longlong2*>(row + s));
          }
          v[s] = x.x;
          v[s + 1] = x.y;
        }
        int64_t P = 0;
#pragma unroll
        for (int s = 0; s < SMAX; ++s) {
          if (s >= S) break;
          dor |= hi32(v[s]);
          P += v[s];
          if (BASE) {
            b0[s] = v[s] > b0[s] ? v[s] : b0[s];
            b1[s] += v[s];
          } else if (P > b0[s]) {
            b0[s] = P;
            br[s] = static_cast<int32_t>(r);
          }
        }
        tor |= hi32(P);
        if (BASE) {
          const uint64_t k = (static_cast<uint64_t>(P) << 16) | static_cast<uint64_t>(65535 - r);
          slow = k > slow ? k : slow;
        }
      }
    }
#pragma unroll
    for (int s = 0; s < SMAX; ++s) {
      if (s >= S) break;
      uint64_t k0;
      if (BASE) k0 = static_cast<uint64_t>(b0[s]);
      else k0 = b0[s] < 0 ? 0ull : (static_cast<uint64_t>(b0[s]) << 16) | static_cast<uint64_t>(65535 - br[s]);
      const uint64_t m0 = warp_max_u64(k0);
      const uint64_t m1 = GAIN   ? warp_max_u64(static_cast<uint64_t>(b1[s]))
                          : BASE ? warp_sum_u64(static_cast<uint64_t>(b1[s]))
                                 : 0;
      if (lane == 0) {
        red[warp][s] = m0;
        red[warp][32 + s] = m1;
      }
    }
    if (BASE) {
      const uint64_t ks = warp_max_u64(slow);
      if (lane == 0) red[warp][64] = ks;
    }
    __syncthreads();
    if (warp == 0) {
      uint64_t v0 = 0, v1 = 0, v2 = 0;
      if (lane < S)
        for (int ww = 0; ww < kGenThreads / 32; ++ww) {
          v0 = red[ww][lane] > v0 ? red[ww][lane] : v0;
          if (BASE) v1 += red[ww][32 + lane];
          else v1 = red[ww][32 + lane] > v1 ? red[ww][32 + lane] : v1;
        }
      if (BASE)
        for (int ww = 0; ww < kGenThreads / 32; ++ww) v2 = red[ww][64] > v2 ? red[ww][64] : v2;
      if (GAIN) finalize_gain(p, S, t, w, v0, static_cast<int64_t>(v1), lane, acc);
      else if (BASE) finalize_base(p, S, t, v0, v1, v2, lane, bacc);
      else finalize_frontier(p, S, t, v0, lane, acc);
    }
    __syncthreads();
    if constexpr (RING) {
      // every thread is done with step t: the chunks wholly before the next
      // step's first byte are free, and each freed stage takes the next chunk
      if (threadIdx.x == 0) {
        const int64_t free_upto = min(nchunks, (s0 + RS8 - A0) >> cshift);
        if (released < free_upto && issued < nchunks) fence_proxy_async_smem();
        for (; released < free_upto; ++released)
          if (issued < nchunks) issue(issued++);
      }
    }
  }
  if constexpr (RING) {
    // copies still in flight (only when a wait gave up): let them land before
    // the CTA's shared memory is released
    if (threadIdx.x == 0)
      for (int64_t c = released; c < issued; ++c)
        mbar_wait_timeout(&full[static_cast<uint32_t>(c) & (NST - 1)], static_cast<uint32_t>(c >> ceil_log2(NST)) & 1u);
  }
  if (BASE && warp == 0) flush_base(p, S, bacc, lane);
  if (!BASE && p.X && warp == 0) flush_window(p, S, acc, lane);
  if (GAIN && p.quality) qual_window(p, qa, -2, lane);
  const uint32_t bits = range_bits(__reduce_or_sync(kFull, dor), __reduce_or_sync(kFull, tor)) |
                        ((RING && *abort) ? SF_ST_TIMEOUT : 0u);
  if (lane == 0) report(p.status, bits);
}

}  // namespace

EncodeFn encode_fn() {
  static EncodeFn fn = [] {
    void* f = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &f, 12000, cudaEnableDefault, &q) !=
            cudaSuccess ||
        q != cudaDriverEntryPointSuccess)
      f = nullptr;
    return reinterpret_cast<EncodeFn>(f);
  }();
  return fn;
}

namespace {

// One lane per (step, stage) instead of tiles: small steps, whose S warp
// reductions each outweigh their few rank rows, and the evidence pass over more
// stages than the tiles take.  A warp walks its steps' ranks one after another, so
// the warps (20 per SM) need steps enough to go round, and a step past 32 bits, walked
// in 64, takes about twice as long where the other forms lose a fifth.  The rank limits
// are where the lanes no longer gain on ordinary steps what half as many long ones
// would lose.  Us, the best other form / lanes, for ordinary steps and, in brackets,
// the same times 64:
//   frontier              48000 x 16 x 6    26.7 / 12.4 (26.7 / 20.5)
//                         48000 x 48 x 6    32.8 / 32.4 (33.0 / 51)
//                         60000 x 97 x 1    22.6 / 16.4 (22.6 / 16.4)
//                         60000 x 129 x 2   33.7 / 37.6 (33.5 / 54)
//                         60000 x 97 x 4    45.1 / 47.0 (45.2 / 67)
//   with window sums      60000 x 65 x 2    39.1 / 18.5 (39.2 / 24.6)
//                         60000 x 97 x 3    49.2 / 38.1 (49.2 / 53)
//                         60000 x 193 x 2     55 / 58   (55 / 86)
//   baselines             60000 x 97 x 3      54 / 37   (54 / 51)
//                         60000 x 193 x 4     86 / 87   (86 / 123)
//                         48000 x 64 x 8      62 / 46   (62 / 79)
//                         24000 x 64 x 16     53 / 46   (53 / 84)
//                         24000 x 48 x 12   39.5 / 36.8 (39.2 / 66)
//   evidence              24000 x 64 x 16     93 / 55   (97 / 109)
//                         24000 x 64 x 8    34.9 / 30.6 (51 / 59)
//                         24000 x 64 x 10     42 / 43   (51 / 85)
//                         608 x 96 x 20     26.7 / 14.3 (27.0 / 29.9), a CTA per step / lanes
//                         608 x 1000 x 20     92 / 110  (92 / 316)
//                         1500 x 1000 x 20   251 / 130  (250 / 374)
//   with quality sums     24000 x 16 x 10     53 / 33.8 (63 / 56)
//                         24000 x 48 x 16    127 / 88   (127 / 164)
//                         24000 x 32 x 12     49 / 65   (49 / 116)
//                         100000 x 100 x 2   188 / 114  (188 / 114)
//                         66666 x 100 x 3    143 / 114  (143 / 186)
//                         33333 x 50 x 3      43 / 43   (43 / 69)
//                         390625 x 64 x 4    506 / 401  (508 / 610)
//                         83333 x 24 x 10    150 / 117  (185 / 202)
//                         97656 x 64 x 16    546 / 428  (573 / 776)
//                         19531 x 64 x 16    119 / 107  (127 / 205)
//                         1790 x 15 x 32     100 / 15   (101 / 25), a CTA per step / lanes
//                         855 x 60 x 20       39 / 25   (39 / 53)
//                         1300 x 96 x 20      57 / 37   (57 / 84)
//                         1300 x 128 x 24     70 / 45   (70 / 107)
//                         1300 x 300 x 24    113 / 97   (113 / 242)
//                         2500 x 192 x 24    131 / 90   (131 / 220)
//                         2500 x 192 x 20    105 / 88   (105 / 214)
//                         9000 x 192 x 20    367 / 251  (368 / 499)
//   medians only 8-byte   10000 x 64 x 6    22.5 / 14.5 (22.6 / 30.8)
//   aligned               5000 x 64 x 4     12.4 / 10.3 (12.3 / 16.5)
//                         20000 x 64 x 6      40 / 54   (40 / 111), with quality sums
bool use_step_lanes(int kind, bool windows, int64_t T, int64_t R, int64_t S, bool fast, int sms) {
  const int64_t tiles = (T + 32 / S - 1) / (32 / S);
  if (tiles < int64_t(sms) * 4) return false;
  if (S > 16) {  // against a CTA per step
    if (kind == kGain) return R <= 192 || T >= int64_t(sms) * (S > 24 ? 4 : 10);
    if (kind != kGainQuality) return false;
    if (R <= (S < 24 ? 40 : 64)) return true;
    if (S >= 24) return T * S >= int64_t(sms) * (R <= 96 ? 120 : R <= 128 ? 150 : 260);
    return R <= 192 && T >= int64_t(sms) * (R <= 64 ? 5 : R <= 96 ? 8 : R <= 128 ? 11 : 50);
  }
  if (!fast)  // against a CTA per step
    return T >= int64_t(sms) * 32 && tiles >= int64_t(sms) * 8 && (kind != kGainQuality || S == 16 || R <= 16);
  const bool full = S <= 4 || S == 8 || S == 16;  // few or none of the lanes idle
  switch (kind) {
    case kFrontier:
      if (lanes_groups(R, S) != 0) return false;
      if (S <= 4) return R <= (S == 1 ? (windows ? 192 : 128) : S == 2 ? (windows ? 128 : 96) : windows ? 100 : 64);
      return R <= (S <= 8 ? 48 : 32) && R * S * 8 <= 3072;
    case kBase: return R <= (S == 1 ? 192 : S <= 3 ? 128 : S == 4 ? 100 : S <= 8 ? 64 : S <= 11 || S == 16 ? 48 : 32);
    case kGain: return R <= (S == 16 ? 128 : full ? 64 : S <= 11 ? 48 : 32);
    default: {
      const int64_t per_sm = tiles / sms;
      if (R <= 16) return true;
      if (S >= 9 && S <= 11) return R <= 24 && per_sm >= 100;
      const bool many = per_sm >= (S <= 2 ? 16 : S == 3 ? 32 : S == 4 ? 64 : 100);
      return full && per_sm >= 16 && R <= (!many || S == 8 ? 48 : S == 16 ? 80 : 128);
    }
  }
}

// A CTA per step (stream_generic_kernel) instead of tiles: few small steps that are not
// whole 128-byte rows, whose tiles' barriers, copies and patched rows cost more than
// plain loads (us, tiles / CTAs: frontier 100 x 614 x 4 6.2 / 4.1, 200 x 171 x 5
// 6.2 / 4.1, 450 x 614 x 1 6.2 / 4.1, 620 x 614 x 1 6.2 / 6.2; evidence 152 x 1000 x 1
// 12.5 / 8.2; baselines 200 x 171 x 12 8.2 / 10.3).
bool use_step_ctas(int kind, int64_t T, int64_t R, int64_t S, bool whole, int sms) {
  return !whole && R * S * 8 <= 20 * 1024 && T <= int64_t(sms) * (S <= 4 ? 3 : 2) && (kind == kFrontier || S <= 8);
}

// Whether the evidence pass keeps whole windows of medians (`rows` 128-byte
// rows each) in shared memory, and how.  Two slots let a window's copy run
// under the steps of the one before; one slot stands idle for a copy at each
// window's end, which sixteen steps repay.  (Beside every tile they double what
// the ring carries: 50000 x 1024 x 10 913 against 807 us, 60000 x 256 x 8 418
// against 262 us, 10000 x 2048 x 4 253 against 126 us.  In regime 0, read through
// L1 by warps that hold whole steps, they were slower in shared memory, 128 x 8 241
// against 180 us.)
void plan_medians(Params& p, int rows) {
  p.m_boxes = (rows + kMaxBoxRows - 1) / kMaxBoxRows;
  p.m_box_rows = ((rows + p.m_boxes - 1) / p.m_boxes + 7) / 8 * 8;  // whole 1024-byte swizzle atoms
  p.m_bytes = p.m_boxes * p.m_box_rows * kRowBytes;
  p.m_slots = p.W < 16 ? 0 : 2 * p.m_bytes <= 72 * 1024 ? 2 : p.m_bytes <= 104 * 1024 ? 1 : 0;
}

// Ranks per tile, at most `most`, for a group of `threads`: the fewest rounds
// of its threads over a step, then the fewest tiles and ranks copied twice.
int64_t choose_tile_ranks(int64_t R, int64_t most, int64_t threads) {
  int64_t best = 0, best_cost = 0;
  const int64_t n0 = (R + most - 1) / most;
  for (int64_t n = n0; n < n0 + 4; ++n)
    for (const int64_t unit : {int64_t(32), threads}) {
      // n even tiles; last, the most whole rounds of the threads that a tile holds
      const int64_t nr = n < n0 + 3 ? std::min(R, ((R + n - 1) / n + unit - 1) / unit * unit) : most / unit * unit;
      if (nr > most || nr == 0 || nr > R) continue;
      const int64_t tiles = (R + nr - 1) / nr, last = R - (tiles - 1) * nr;
      const int64_t rounds = (tiles - 1) * ((nr + threads - 1) / threads) + (last + threads - 1) / threads;
      const int64_t cost = rounds * threads + 64 * tiles + (tiles * nr - R) / 2;
      if (best == 0 || cost < best_cost) {
        best = nr;
        best_cost = cost;
      }
    }
  return best;
}

}  // namespace

cudaError_t launch_stream_pass(const StreamJob& j, cudaStream_t stream) {
  Params p{};
  p.T = j.T;
  p.R = j.R;
  p.S = j.S;
  p.a = j.a;
  p.lead = j.lead;
  p.mk = j.mk;
  p.X = j.X;
  p.D = j.D;
  p.E = j.E;
  p.C = j.C;
  p.step_lead = j.step_lead;
  p.t0 = j.t0;
  p.W = j.W;
  p.w_first = j.t0 / j.W;
  p.m = j.m;
  p.wall = j.wall;
  p.other_stage = j.other_stage;
  p.eta_num = j.eta_num;
  p.eta_den = j.eta_den;
  p.Y = j.Y;
  p.quality = j.quality;
  p.status = j.status;
  p.d = j.d;
  p.bM = j.bM;
  p.bSUM = j.bSUM;
  p.bSLOW = j.bSLOW;
  p.bRANK0 = j.bRANK0;

  const int64_t RS = j.R * j.S;
  const int64_t rows = j.T * RS / 16;  // whole 128-byte rows of d
  const bool fast = j.S <= 16 && rows >= 1 && rows <= int64_t(0x7fffffff) && encode_fn() != nullptr &&
                    (!j.gain || reinterpret_cast<uintptr_t>(j.m) % 16 == 0);
  const int sms = sm_count();
  // few steps over many ranks (frontier and aggregation): split each step's
  // ranks over a cluster so that every SM streams
  if (const Split q = plan_split(j, sms); q.csize > 0) {
    auto go = [&](int csize) {
      const int S = static_cast<int>(j.S);
      return q.rows == 4 ? dispatch_split<4>(S, j.d, p, csize, stream, j.after_clear)
                         : dispatch_split<2>(S, j.d, p, csize, stream, j.after_clear);
    };
    count_launch();
    cudaError_t e = go(q.csize);
    if (e != cudaSuccess && q.csize > 8) {  // a 16-CTA cluster that cannot be placed: portable size
      cudaGetLastError();
      e = go(8);
    }
    return e;
  }
  const int kind = j.gain ? (j.quality ? kGainQuality : kGain) : j.base ? kBase : kFrontier;
  if (use_step_lanes(kind, j.X != nullptr, j.T, j.R, j.S, fast, sms)) {
    count_launch();
    return launch_step_lanes(kind, p, stream, j.after_clear);
  }
  const bool whole = RS % 16 == 0 && j.S % 2 == 0;
  if (fast && !use_step_ctas(kind, j.T, j.R, j.S, whole, sms)) {
    const bool gain = j.gain;
    const int warps = consumer_warps(kind, j.S);
    // elements a tile may hold before its first one, in the 128-byte row both share
    const int64_t pad = whole ? 0 : 15;
    p.rows = rows;
    auto box_for = [&](int64_t elems) { return (pad + elems + 15) / 16; };
    // frontier and aggregation over small steps: several steps per warp instruction
    const int lanes = kind == kFrontier ? lanes_groups(j.R, j.S) : 0;
    const int64_t r0_rows = r0_stage_bytes(kind, j.S) / kRowBytes;
    p.regime = box_for(RS) <= r0_rows ? 0 : 1;
    p.m_rows = gain ? (j.T + j.W - 1) / j.W * RS / 16 : 0;
    if (p.m_rows >= 1 && p.regime == 1 && j.T >= int64_t(sms) * 4) plan_medians(p, static_cast<int>(box_for(RS)));
    p.ring_bytes = gain && p.regime == 1 ? kGainBytes : kRingBytes;
    if (p.regime == 0) {
      // whole steps per tile: as many as fit, fewer where that would leave warps without a tile
      const int64_t unit = lanes > 0 ? lanes : 1;  // whole rounds of G steps
      int64_t K = std::max<int64_t>(unit, (r0_rows * 16 - pad) / RS / unit * unit);
      const int64_t share = (j.T + int64_t(sms) * warps - 1) / (int64_t(sms) * warps);
      K = std::min(K, (share + unit - 1) / unit * unit);
      p.K = static_cast<int>(K);
      p.box_rows = static_cast<int>(box_for(K * RS));
      p.nst = 2 * warps;
      p.stage_bytes = r0_stage_bytes(kind, j.S);
      p.groups = 1;
    } else {
      // Warp groups take the steps in turn, so that the reductions of several
      // small steps are in flight; each group owns its ring stages: a stage is
      // refilled only after its own group has consumed it, so no wait can pass
      // a phase early.
      // Four groups up to 64 KB (evidence: 32 KB, where its warps are fewer per
      // byte), two up to 128 KB: baselines 512 x 12 with two groups 174 us, four 152;
      // 1003 x 16 with one 111, two 89; evidence 1001 x 8 with two 81 us, four 114.
      const int64_t kb = 1024, step_bytes = RS * 8;
      if (!gain) p.groups = step_bytes <= 64 * kb ? 4 : step_bytes <= 128 * kb ? 2 : 1;
      else p.groups = step_bytes <= 32 * kb ? 4 : step_bytes <= 128 * kb ? 2 : 1;
      while (p.groups > 1 && (p.groups - 1) * int64_t(sms) >= j.T) p.groups /= 2;  // a group for every step of a CTA
      const int64_t threads = warps * 32 / p.groups;  // of a group
      // tiles that leave each group three stages
      const int64_t ring = p.ring_bytes - p.m_slots * p.m_bytes;
      p.m_by_tma = gain && !p.m_slots ? 1 : 0;
      const int64_t fit = ring / ((p.m_by_tma ? 2 : 1) * 3 * p.groups * kRowBytes) / 8 * 8;  // rows
      const int64_t max_rows = std::min<int64_t>(kMaxBoxRows, gain ? fit : p.groups == 4 ? kMaxBoxRows / 2 : kMaxBoxRows);
      p.tile_ranks = static_cast<int>(choose_tile_ranks(j.R, std::max<int64_t>(32, (max_rows * 16 - pad) / j.S / 32 * 32), threads));
      p.tiles_per_step = static_cast<int>((j.R + p.tile_ranks - 1) / p.tile_ranks);
      p.box_rows = static_cast<int>(box_for(int64_t(p.tile_ranks) * j.S));
      p.stage_bytes = (p.box_rows * kRowBytes + 1023) / 1024 * 1024 * (p.m_by_tma ? 2 : 1);
      // frontier and baselines: more copies in flight than these read slower (8192 x 8
      // frontier: 1423 us with four stages, 1569 us with the six that fit)
      const int most_stages = (gain ? 8 : p.groups == 1 ? 4 : 3) * p.groups;
      p.nst = static_cast<int>(std::min<int64_t>({ring / p.stage_bytes, most_stages, kMaxStages}) / p.groups * p.groups);
    }
    const bool swz = j.S == 4 || j.S == 8 || j.S == 16 || lanes > 0;
    auto encode = [&](CUtensorMap* out, const int64_t* base, int64_t nrows, int box_rows) {
      const cuuint64_t gdim[2] = {16, static_cast<cuuint64_t>(nrows)};
      const cuuint64_t gstride[1] = {kRowBytes};
      const cuuint32_t box[2] = {16, static_cast<cuuint32_t>(box_rows)};
      const cuuint32_t estride[2] = {1, 1};
      return encode_fn()(out, CU_TENSOR_MAP_DATA_TYPE_INT64, 2, const_cast<int64_t*>(base), gdim, gstride, box,
                         estride, CU_TENSOR_MAP_INTERLEAVE_NONE,
                         swz ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_NONE,
                         CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    };
    CUtensorMap map, map_m;
    if (encode(&map, j.d, rows, p.box_rows) != CUDA_SUCCESS) return cudaErrorInvalidValue;
    map_m = map;
    if (p.m_by_tma || p.m_slots) {
      if (p.m_rows > int64_t(0x7fffffff) ||
          encode(&map_m, j.m, p.m_rows, p.m_slots ? p.m_box_rows : p.box_rows) != CUDA_SUCCESS)
        return cudaErrorInvalidValue;
    }
    const int64_t units = p.regime == 0 ? (j.T + p.K - 1) / p.K : j.T;
    const int grid = static_cast<int>(std::min<int64_t>(sms, units));
    count_launch();
    const bool pdl = j.after_clear;
    if (lanes > 0) return launch_lanes(lanes, map, p, grid, stream, pdl);
    TiledLaunch* const launch = kind == kGain          ? (whole ? launch_gain_aligned : launch_gain_unaligned)
                                : kind == kGainQuality ? (whole ? launch_quality_aligned : launch_quality_unaligned)
                                : kind == kBase        ? (whole ? launch_base_aligned : launch_base_unaligned)
                                                       : (whole ? launch_frontier_aligned : launch_frontier_unaligned);
    return launch(map, map_m, p, grid, stream, pdl);
  }
  count_launch();
  const bool vec = j.S % 2 == 0;  // whole-row 16-byte loads (frontier and baseline passes)
  // bulk-copy ring: the smallest power-of-two chunk (4-16 KB) of which
  // kGenRingStages - 1 hold a whole step; larger steps read global memory
  const int64_t step_bytes = j.R * j.S * 8;
  uint32_t chunk = 0;
  for (uint32_t c = 4096; c <= 16384 && !chunk; c *= 2)
    if (step_bytes <= int64_t(kGenRingStages - 1) * c) chunk = c;
  p.stage_bytes = static_cast<int>(chunk);
  p.nst = static_cast<int>(kGenRingStages);
  auto generic = [&](auto smax) {
    constexpr int SM = decltype(smax)::value;
    const bool pdl = j.after_clear;
    auto go = [&](auto kern, bool ring) {
      const size_t smem = ring ? size_t(kGenRingStages) * chunk : 0;
      int per_sm = 4;
      if (ring) {
        cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             static_cast<int>(smem));
        if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kGenThreads, smem);
        if (e != cudaSuccess) return e;
        per_sm = std::max(per_sm, 1);
      }
      const int grid = static_cast<int>(std::min<int64_t>(int64_t(sms) * per_sm, j.T));
      return launch_ex(kern, grid, kGenThreads, smem, stream, pdl, j.d, p);
    };
    if constexpr (SM > 16) {
      // more than 16 stages: registers hold these kernels to one or two CTAs
      // per SM, and the bulk-copy ring keeps the loads off their step chain
      // (512 x 24: 0.434 -> 0.405 ms).  Up to 16 stages these kernels see few
      // steps, and four CTAs per SM hide the loads.
      if (chunk != 0) {
        if (j.gain) return go(stream_generic_kernel<SM, 1, false, true>, true);
        if (j.base && vec) return go(stream_generic_kernel<SM, 2, true, true>, true);
        if (j.base) return go(stream_generic_kernel<SM, 2, false, true>, true);
        if (vec) return go(stream_generic_kernel<SM, 0, true, true>, true);
        return go(stream_generic_kernel<SM, 0, false, true>, true);
      }
    }
    if (j.gain) return go(stream_generic_kernel<SM, 1, false, false>, false);
    if (j.base && vec) return go(stream_generic_kernel<SM, 2, true, false>, false);
    if (j.base) return go(stream_generic_kernel<SM, 2, false, false>, false);
    if (vec) return go(stream_generic_kernel<SM, 0, true, false>, false);
    return go(stream_generic_kernel<SM, 0, false, false>, false);
  };
  if (j.S <= 4) return generic(std::integral_constant<int, 4>{});
  if (j.S <= 8) return generic(std::integral_constant<int, 8>{});
  if (j.S <= 16) return generic(std::integral_constant<int, 16>{});
  return generic(std::integral_constant<int, 32>{});
}

}  // namespace sf