// sf_tiled_base_aligned.cu - the tiled routing-baseline pass, steps of whole 128-byte rows.
#include "sf_tiled.cuh"

namespace sf {

cudaError_t launch_base_aligned(const CUtensorMap& map, const CUtensorMap& map_m, const Params& p, int grid,
                                cudaStream_t stream, bool pdl) {
  return dispatch_tiled<kBase, true>(map, map_m, p, grid, stream, pdl);
}

}  // namespace sf
