// sf_ingest.cu - rank-major ingest.  The window-boundary gather of Sec. 5
// delivers each window as one [R][n][S] block (every rank's [n, S] buffer in
// rank order); the kernels of this library read steps as [T][R][S].  The
// conversion is a pure copy: each thread moves 16 bytes (8 when S is odd)
// of one destination row, so a warp writes 512 contiguous bytes while its
// reads are whole S*8-byte stage vectors of consecutive ranks.
#include <algorithm>
#include <cstdint>

#include "sf_device.cuh"
#include "sf_launch.h"

namespace sf {
namespace {

constexpr int kIngThreads = 256;

// dst[t][r][s] = src block b = t / N, [r][t - b*N][s]; block b starts at
// element b*R*N*S and holds n_b = min(N, T - b*N) steps.  A CTA fills one
// destination step at a time, with PARTS one of `parts` pieces of a step: few
// steps of many ranks then have eight CTAs per SM (us: 1 x 8192 x 8 19.4 -> 6.3,
// 100 x 8192 x 8 51 -> 20, 250 x 8192 x 8 66 -> 46, 100 x 30000 x 16 347 -> 129).
// One kernel for both forms read slower over many steps (100000 x 128 x 8 263 -> 401).
template <int kUnit, bool PARTS>  // kUnit int64 values moved per thread: 2 (S even) or 1
__global__ void __launch_bounds__(kIngThreads) gathered_to_steps_kernel(const int64_t* __restrict__ src, int64_t T,
                                                                        int64_t R, int64_t S, int64_t N,
                                                                        int parts, int64_t* __restrict__ dst) {
  const int units = static_cast<int>(R * S / kUnit);  // per destination step (<= 2^21)
  const int su = static_cast<int>(S / kUnit);
  const int64_t pieces = PARTS ? T * parts : T;
  for (int64_t id = blockIdx.x; id < pieces; id += gridDim.x) {
    int64_t t = id;
    int begin = 0, end = units;
    if constexpr (PARTS) {
      t = id / parts;
      const int part = static_cast<int>(id - t * parts);
      begin = static_cast<int>(int64_t(units) * part / parts);
      end = static_cast<int>(int64_t(units) * (part + 1) / parts);
    }
    const int64_t b = t / N, tl = t - b * N;
    const int64_t nb = T - b * N < N ? T - b * N : N;
    const int64_t* sb = src + b * R * N * S + tl * S;
    int64_t* dt = dst + t * R * S;
#pragma unroll 4
    for (int j = begin + threadIdx.x; j < end; j += kIngThreads) {
      const int r = j / su;
      const int s = (j - r * su) * kUnit;
      const int64_t* from = sb + int64_t(r) * nb * S + s;
      if constexpr (kUnit == 2)
        *reinterpret_cast<longlong2*>(dt + 2 * int64_t(j)) = __ldg(reinterpret_cast<const longlong2*>(from));
      else
        dt[j] = __ldg(from);
    }
  }
}

// Through shared memory: tiles of kTileSteps steps of one window by as many
// ranks as fit, so that both sides move in runs (a rank's kTileSteps S values in,
// a step's ranks x S values out) where the kernel above reads S values at a time
// and gives a whole CTA to a step.  A warp moves one run at a time, 8 bytes a lane
// (16 bytes a lane read slower: fewer lanes per run, more registers).
constexpr int kTileSteps = 16;
constexpr int kTileBytes = 48 * 1024;

// values of a rank's run in the tile, padded to an odd number against bank conflicts
__host__ __device__ constexpr int tile_pitch(int S) { return kTileSteps * S | 1; }

struct IngestTiles {
  int ranks = 0;      // of a tile; 0: no tiles
  int64_t count = 0;
};

// Steps a CTA has little to do for, and tiles for every SM (us, directly / tiles:
// 100000 x 16 x 8 102.6 / 44.8, 100000 x 31 x 7 160 / 90, 20000 x 64 x 5 53.5 / 27.3;
// 1500 x 32 x 6, of 94 tiles, 4.1 / 6.2; 3000 x 120 x 3, of 188, 8.2 / 10.3; 4000 x 40 x 7, of
// 250, 10.3 / 8.2; 3000 x 4 x 1 6.2 / 4.1; 5000 x 128 x 1 8.2 / 10.3, 24000 26.7 / 22.6).  Odd
// stage counts, moved 8 bytes at a time directly, gain up to 3 KB a step; even ones, moved
// 16 bytes, up to 2.5 KB and 64 ranks (100000 x 64 x 4 117 / 101, 96 x 4 130 / 150, 32 x 12
// 125 / 122, 128 x 2 117 / 143).
IngestTiles plan_tiles(int64_t T, int64_t R, int64_t S, int64_t N) {
  IngestTiles p;
  const bool small = S % 2 == 0 ? R <= 64 && R * S <= 320 : R <= 128 && R * S <= 384;
  if (N < kTileSteps || !small) return p;
  // even shares of the ranks (100000 x 64 x 6, whose tiles hold 63 ranks: 63 and 1 206 us, 32 and 32 125)
  const int64_t most = kTileBytes / (8 * tile_pitch(static_cast<int>(S))), blocks = (R + most - 1) / most;
  p.count = (T + N - 1) / N * ((N + kTileSteps - 1) / kTileSteps) * blocks;
  const int halves = R * S <= 64 ? 2 : S == 1 && R > 96 ? 10 : 3;  // half tiles per SM
  if (2 * p.count >= sm_count() * halves) p.ranks = static_cast<int>((R + blocks - 1) / blocks);
  return p;
}

__global__ void __launch_bounds__(kIngThreads) gathered_tiles_kernel(const int64_t* __restrict__ src, int64_t T,
                                                                     int64_t R, int S, int64_t N, int ranks,
                                                                     int64_t* __restrict__ dst) {
  __shared__ int64_t tile[kTileBytes / 8];  // [ranks][pitch]
  constexpr int kWarps = kIngThreads / 32;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int pitch = tile_pitch(S);
  const int step_r = 32 / S, step_s = 32 - step_r * S;  // a lane's next value of a step: ranks on, stages on
  const int64_t per_window = (N + kTileSteps - 1) / kTileSteps, windows = (T + N - 1) / N;
  const int64_t blocks = (R + ranks - 1) / ranks, tiles = windows * per_window * blocks;
  for (int64_t id = blockIdx.x; id < tiles; id += gridDim.x) {
    const int64_t b = id % blocks, q = id / blocks;
    const int64_t win = q / per_window, t0 = (q - win * per_window) * kTileSteps;
    const int64_t nb = min(N, T - win * N);
    if (t0 >= nb) continue;  // the last window may be short
    const int steps = static_cast<int>(min(int64_t(kTileSteps), nb - t0));
    const int64_t r0 = b * ranks;
    const int nr = static_cast<int>(min(int64_t(ranks), R - r0));
    const int64_t* from = src + win * N * R * S + (r0 * nb + t0) * S;
    const int run = steps * S;
#pragma unroll 4
    for (int r = warp; r < nr; r += kWarps)
      for (int i = lane; i < run; i += 32) tile[r * pitch + i] = __ldg(from + r * nb * S + i);
    __syncthreads();
    int64_t* to = dst + ((win * N + t0) * R + r0) * S;
    for (int t = warp; t < steps; t += kWarps) {
      int r = lane / S, s = lane - r * S;
#pragma unroll 4
      for (int i = lane; i < nr * S; i += 32) {
        to[t * R * S + i] = tile[r * pitch + t * S + s];
        r += step_r;
        s += step_s;
        if (s >= S) {
          s -= S;
          ++r;
        }
      }
    }
    __syncthreads();
  }
}

}  // namespace

cudaError_t launch_gathered_to_steps(const int64_t* src, int64_t T, int64_t R, int64_t S, int64_t N, int64_t* dst,
                                     cudaStream_t stream) {
  N = std::min(N, T);  // one window holds them all
  if (const IngestTiles tiles = plan_tiles(T, R, S, N); tiles.ranks > 0) {
    const int grid = static_cast<int>(std::min<int64_t>(tiles.count, int64_t(sm_count()) * 4));
    count_launch();
    gathered_tiles_kernel<<<grid, kIngThreads, 0, stream>>>(src, T, R, static_cast<int>(S), N, tiles.ranks, dst);
    return cudaGetLastError();
  }
  const int unit = S % 2 == 0 ? 2 : 1;
  const int64_t slots = int64_t(sm_count()) * 8;
  const int parts = static_cast<int>(std::min(slots / T, R * S / (4096 * unit)));  // at least 4096 units each
  const int grid = static_cast<int>(std::min(T * std::max(parts, 1), slots));
  count_launch();
  auto go = [&](auto kern) { kern<<<grid, kIngThreads, 0, stream>>>(src, T, R, S, N, parts, dst); };
  if (unit == 2) parts > 1 ? go(gathered_to_steps_kernel<2, true>) : go(gathered_to_steps_kernel<2, false>);
  else parts > 1 ? go(gathered_to_steps_kernel<1, true>) : go(gathered_to_steps_kernel<1, false>);
  return cudaGetLastError();
}

}  // namespace sf
