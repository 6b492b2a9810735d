// sf_tiled_quality_unaligned.cu - the tiled evidence pass with telemetry-quality sums, steps that are not whole 128-byte rows.
#include "sf_tiled.cuh"

namespace sf {

cudaError_t launch_quality_unaligned(const CUtensorMap& map, const CUtensorMap& map_m, const Params& p, int grid,
                                     cudaStream_t stream, bool pdl) {
  return dispatch_tiled<kGainQuality, false>(map, map_m, p, grid, stream, pdl);
}

}  // namespace sf
