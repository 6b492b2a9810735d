// sf_tiled_gain_unaligned.cu - the tiled evidence pass, steps that are not whole 128-byte rows.
#include "sf_tiled.cuh"

namespace sf {

cudaError_t launch_gain_unaligned(const CUtensorMap& map, const CUtensorMap& map_m, const Params& p, int grid,
                                  cudaStream_t stream, bool pdl) {
  return dispatch_tiled<kGain, false>(map, map_m, p, grid, stream, pdl);
}

}  // namespace sf
