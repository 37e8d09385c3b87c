// Bins-fastest slice kernels of spreading widths 7 and 8.
#include "slice_tiles_dispatch.cuh"

namespace aahrt {

template cudaError_t tile_width<7>(const TileCall &, const TileArgs &, const float2 *, float2 *);
template cudaError_t tile_width<8>(const TileCall &, const TileArgs &, const float2 *, float2 *);

}  // namespace aahrt
