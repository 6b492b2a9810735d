// sf_tiled_quality_aligned.cu - the tiled evidence pass with telemetry-quality sums, steps of whole 128-byte rows.
#include "sf_tiled.cuh"

namespace sf {

cudaError_t launch_quality_aligned(const CUtensorMap& map, const CUtensorMap& map_m, const Params& p, int grid,
                                   cudaStream_t stream, bool pdl) {
  return dispatch_tiled<kGainQuality, true>(map, map_m, p, grid, stream, pdl);
}

}  // namespace sf
