// sf_tiled_base_unaligned.cu - the tiled routing-baseline pass, steps that are not whole 128-byte rows.
#include "sf_tiled.cuh"

namespace sf {

cudaError_t launch_base_unaligned(const CUtensorMap& map, const CUtensorMap& map_m, const Params& p, int grid,
                                  cudaStream_t stream, bool pdl) {
  return dispatch_tiled<kBase, false>(map, map_m, p, grid, stream, pdl);
}

}  // namespace sf
