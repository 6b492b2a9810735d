// sf_lanes.cu - the tiled frontier and window aggregation pass over small
// steps, several to a warp instruction.
#include "sf_tiled.cuh"

namespace sf {

namespace {

constexpr int kLaneWarps = consumer_warps(kFrontier, 1);

// --------------------------------------------------------------------------
// Frontier pass over small steps (R*S <= 768, S in {2, 4, 8, 16}): G steps
// share each warp instruction.  A warp splits into G groups of L = 32 / G
// lanes; group g takes step kk0 + g of the warp's tile and lane j of the group
// visits ranks j, j + L, ... in increasing order, so a strict '>' keeps the
// lowest rank within a lane.  The per-stage packed keys (F << 16 | 65535 - r)
// are then reduced over the group's L lanes by exchanges that halve the set of
// keys a lane holds at each step (G steps' reductions in the instructions of
// one), and the lanes j < S of each group run the step's epilogue for their
// own step, so the per-step epilogue cost is shared by G steps as well.  The
// tiles (K whole steps, K a multiple of G) arrive through the same warp-owned
// ring stages as the other small-step path, from the same producer.  With
// consecutive ranks in consecutive lanes, the 128-byte swizzle places the 16
// or 8 lanes of a group on distinct 16-byte bank groups, so a group's row
// reads are conflict free.
template <int S, int L>
__device__ __forceinline__ uint64_t group_max_keys(uint64_t (&k)[S], int j) {
  static_assert(L >= S && (S & (S - 1)) == 0 && (L & (L - 1)) == 0, "L >= S, both powers of two");
#pragma unroll
  for (int lvl = 0; (L >> (lvl + 1)) >= 1; ++lvl) {
    const int o = L >> (lvl + 1);
    const int n = S >> lvl;  // keys this lane still holds
    if (n > 1) {
      // the lane with bit o set keeps the upper half of its keys, its partner the lower
      const bool up = (j & o) != 0;
#pragma unroll
      for (int i = 0; i < n / 2; ++i) {
        const uint64_t send = up ? k[i] : k[i + n / 2];
        const uint64_t keep = up ? k[i + n / 2] : k[i];
        const uint64_t got = __shfl_xor_sync(kFull, send, o);
        k[i] = keep > got ? keep : got;
      }
    } else {
      const uint64_t got = __shfl_xor_sync(kFull, k[0], o);
      k[0] = k[0] > got ? k[0] : got;
    }
  }
  // lane j now holds the group maximum of stage j >> (log2 L - log2 S)
  return k[0];
}

// Frontier epilogue of one group's step t (the group's lanes j < S hold the
// packed keys of stages j); the whole warp calls it, live = false for groups
// past the tile's last step.
template <int S, int L>
__device__ __forceinline__ void finalize_group(const Params& p, int64_t t, uint64_t key, int j, bool live,
                                               WinAcc& acc) {
  const bool valid = live && j < S;
  const int64_t F = valid ? static_cast<int64_t>(key >> 16) : 0;
  const int32_t ld = valid ? 65535 - static_cast<int32_t>(key & 0xffffu) : 0;
  int64_t Fprev = __shfl_up_sync(kFull, F, 1, L);
  if (j == 0) Fprev = 0;  // F[t,-1] = 0
  const int64_t a = valid ? F - Fprev : 0;
  const int64_t mk = __shfl_sync(kFull, F, S - 1, L);
  uint64_t km = 0;
  if (p.X && p.step_lead) {
    // leading stage: largest increment, lowest stage on ties
    km = valid ? ((static_cast<uint64_t>(a) << 5) | static_cast<uint64_t>(31 - j)) : 0;
#pragma unroll
    for (int o = 1; o < S; o <<= 1) {
      const uint64_t got = __shfl_xor_sync(kFull, km, o);
      km = km > got ? km : got;
    }
  }
  if (!live) return;
  if (valid) {
    if (p.a) p.a[t * S + j] = a;
    if (p.lead) p.lead[t * S + j] = ld;
  }
  if (j == 0 && p.mk) p.mk[t] = mk;
  if (p.X) {
    const int64_t w = acc.wt.at(t, p.t0, p.W, p.w_first);
    if (w != acc.cur) {
      flush_window(p, S, acc, j);
      acc.cur = w;
      acc.erow = (w * S + j) * p.R;
    }
    acc.x += a;
    acc.dsum += mk;
    if (valid && ld >= 0 && ld < p.R) {  // always true for valid input; guards flagged input
      const int64_t idx = acc.erow + ld;
      if (p.E && a != 0)
        atomicAdd(reinterpret_cast<unsigned long long*>(&p.E[idx]), static_cast<unsigned long long>(a));
      if (p.C) atomicAdd(&p.C[idx], 1);
    }
    if (p.step_lead && j == 0) p.step_lead[t] = static_cast<uint8_t>(31 - static_cast<int>(km & 31u));
  }
}

template <int S, int G>
__global__ void __launch_bounds__((kLaneWarps + kProducers) * 32, 1)
    lanes_kernel(const __grid_constant__ CUtensorMap map, const Params p) {
  constexpr int L = 32 / G;
  constexpr int U = S <= 8 ? 4 : 2;  // rank rows in flight per lane
  constexpr int kShift = ceil_log2(L) - ceil_log2(S);
  extern __shared__ unsigned char smem_raw[];
  unsigned char* ring = align_1024(smem_raw);
  uint64_t* full = reinterpret_cast<uint64_t*>(ring + kRingBytes);
  uint64_t* empty = full + kMaxStages;
  volatile int* abort = reinterpret_cast<volatile int*>(empty + kMaxStages);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t NB = gridDim.x, b = blockIdx.x;
  const int64_t t_begin = p.T * b / NB, t_end = p.T * (b + 1) / NB;

  if (threadIdx.x < kMaxStages) {
    mbar_init(&full[threadIdx.x], 1);
    mbar_init(&empty[threadIdx.x], 1);
    if (threadIdx.x == 0) *abort = 0;
    fence_barrier_init();
  }
  __syncthreads();

  if (warp >= kLaneWarps) {
    if (lane == 0) produce<kLaneWarps>(warp - kLaneWarps, &map, &map, p, t_begin, t_end, ring, full, empty, MedianSlots{}, abort);
    return;
  }
  griddep_wait();  // outputs cleared by the launch before this one (when it is its dependent)

  const int g = lane / L, j = lane % L;
  uint32_t dor = 0, tor = 0;
  WinAcc acc;
  const int R = static_cast<int>(p.R);
  const int64_t n_local = t_end - t_begin;
  const int64_t n_tiles = (n_local + p.K - 1) / p.K;
  // one round: group g takes step kk of `tile` (step t of the pass)
  auto round = [&](const unsigned char* tile, int kk, int64_t t, bool live, bool have) {
    FrontierRows<S> rs;
    rs.init();
    if (have && live) {
      const int q0 = kk * R;
      for (int r0 = j; r0 < R; r0 += L * U) {
        int64_t v[U][S];
#pragma unroll
        for (int u = 0; u < U; ++u)
          if (r0 + L * u < R) load_row<S, true>(tile, 0, q0 + r0 + L * u, v[u]);
#pragma unroll
        for (int u = 0; u < U; ++u)
          if (r0 + L * u < R) rs.row(v[u], r0 + L * u, dor, tor);
      }
    }
    uint64_t k[S];
#pragma unroll
    for (int s = 0; s < S; ++s) k[s] = rs.key(s);
    const uint64_t ks = group_max_keys<S, L>(k, j);
    // lane j < S of the group takes stage j's key from the lane holding it
    const uint64_t mykey = __shfl_sync(kFull, ks, (j & (S - 1)) << kShift, L);
    finalize_group<S, L>(p, t, mykey, j, live, acc);
  };
  // K steps per tile (a multiple of G): the warp's tiles one at a time, G steps per round
  uint32_t i = 0;
  for (int64_t jt = warp; jt < n_tiles; jt += kLaneWarps, ++i) {
    const uint32_t st = 2u * warp + (i & 1u), ph = (i >> 1) & 1u;
    const bool have = mbar_wait_bounded(&full[st], ph, abort);
    const unsigned char* tile = ring + size_t(st) * p.stage_bytes;
    const int nsteps = static_cast<int>(min(int64_t(p.K), n_local - jt * p.K));
    for (int kk0 = 0; kk0 < nsteps; kk0 += G) {
      const int kk = kk0 + g;
      round(tile, kk, t_begin + jt * p.K + kk, kk < nsteps, have);
    }
    __syncwarp();
    if (lane == 0) mbar_arrive(&empty[st]);
  }

  if (p.X) flush_window(p, S, acc, j);
  const uint32_t bits = range_bits(__reduce_or_sync(kFull, dor), __reduce_or_sync(kFull, tor)) |
                        (*abort ? SF_ST_TIMEOUT : 0u);
  if (lane == 0) report(p.status, bits);
}

}  // namespace

// Steps per warp instruction of the small-step frontier pass: the largest
// G in {2, 4, 8} with L = 32 / G >= S and G whole steps in one ring stage;
// 0 when the shape takes the one-step-per-warp path.  (Steps of 6-12 KB,
// one per stage, stay there: a warp taking both of its stages in one round
// has no copy of its own in flight, and the in-order producer then holds
// every warp up; measured at less than half the one-step-per-warp rate.)
int lanes_groups(int64_t R, int64_t S) {
  if (S != 2 && S != 4 && S != 8 && S != 16) return 0;
  if (R * S % 16 != 0) return 0;
  const int64_t step_rows = R * S / 16, max_rows = r0_stage_bytes(kFrontier, S) / kRowBytes;
  int G = 0;
  for (int c = 2; c <= 8; c *= 2)
    if (32 / c >= S && c * step_rows <= max_rows) G = c;
  return G;
}

cudaError_t launch_lanes(int G, const CUtensorMap& map, const Params& p, int grid, cudaStream_t stream, bool pdl) {
#define SF_LANES(SV, GV)                                                                          \
  if (p.S == SV && G == GV) {                                                                       \
    cudaError_t e = cudaFuncSetAttribute(lanes_kernel<SV, GV>, cudaFuncAttributeMaxDynamicSharedMemorySize, \
                                         static_cast<int>(tiled_smem(kFrontier, SV, kRingBytes)));                          \
    if (e != cudaSuccess) return e;                                                               \
    return launch_ex(lanes_kernel<SV, GV>, grid, (kLaneWarps + kProducers) * 32, tiled_smem(kFrontier, SV, kRingBytes), stream, pdl, map, p);   \
  }
  SF_LANES(2, 2)
  SF_LANES(2, 4)
  SF_LANES(2, 8)
  SF_LANES(4, 2)
  SF_LANES(4, 4)
  SF_LANES(4, 8)
  SF_LANES(8, 2)
  SF_LANES(8, 4)
  SF_LANES(16, 2)
#undef SF_LANES
  return cudaErrorInvalidValue;
}

}  // namespace sf
