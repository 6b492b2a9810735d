// sf_tiled_frontier_aligned.cu - the tiled frontier and window aggregation pass, steps of whole 128-byte rows.
#include "sf_tiled.cuh"

namespace sf {

cudaError_t launch_frontier_aligned(const CUtensorMap& map, const CUtensorMap& map_m, const Params& p, int grid,
                                    cudaStream_t stream, bool pdl) {
  return dispatch_tiled<kFrontier, true>(map, map_m, p, grid, stream, pdl);
}

}  // namespace sf
