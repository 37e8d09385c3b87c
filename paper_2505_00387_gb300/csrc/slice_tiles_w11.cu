// Bins-fastest slice kernels of spreading widths 11 and 12.
#include "slice_tiles_dispatch.cuh"

namespace aahrt {

template cudaError_t tile_width<11>(const TileCall &, const TileArgs &, const float2 *, float2 *);
template cudaError_t tile_width<12>(const TileCall &, const TileArgs &, const float2 *, float2 *);

}  // namespace aahrt
