// Bins-fastest slice kernels of spreading widths 2 and 4.
#include "slice_tiles_dispatch.cuh"

namespace aahrt {

template cudaError_t tile_width<2>(const TileCall &, const TileArgs &, const float2 *, float2 *);
template cudaError_t tile_width<4>(const TileCall &, const TileArgs &, const float2 *, float2 *);

}  // namespace aahrt
