// Bins-fastest slice kernels of spreading widths 5 and 6.
#include "slice_tiles_dispatch.cuh"

namespace aahrt {

template cudaError_t tile_width<5>(const TileCall &, const TileArgs &, const float2 *, float2 *);
template cudaError_t tile_width<6>(const TileCall &, const TileArgs &, const float2 *, float2 *);

}  // namespace aahrt
