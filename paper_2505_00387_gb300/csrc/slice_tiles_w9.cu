// Bins-fastest slice kernels of spreading widths 9 and 10.
#include "slice_tiles_dispatch.cuh"

namespace aahrt {

template cudaError_t tile_width<9>(const TileCall &, const TileArgs &, const float2 *, float2 *);
template cudaError_t tile_width<10>(const TileCall &, const TileArgs &, const float2 *, float2 *);

}  // namespace aahrt
