// sf_tiled_frontier_unaligned.cu - the tiled frontier and window aggregation pass, steps that are not whole 128-byte rows.
#include "sf_tiled.cuh"

namespace sf {

cudaError_t launch_frontier_unaligned(const CUtensorMap& map, const CUtensorMap& map_m, const Params& p, int grid,
                                      cudaStream_t stream, bool pdl) {
  return dispatch_tiled<kFrontier, false>(map, map_m, p, grid, stream, pdl);
}

}  // namespace sf
