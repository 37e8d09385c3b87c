// The bins-fastest slice kernels of one spreading width (slice_tiles.cuh)
// behind one function, compiled in separate files so they build in parallel.
//
// Tiles of 32 bins where two grids of nos points leave room for three blocks
// per SM (nos <= 128), of 16 bins for 256 points (and for small plans, whose
// work items would not fill the SMs), of 8 for 512 points: half the traces of a
// pair conflict then, but three blocks share an SM (595 / 756 us forward /
// adjoint of the 8000-trace gather against 677 / 882 with 16 bins and one block
// of 512 threads).
#pragma once

#include "slice_tiles.cuh"

namespace aahrt {

struct TileCall {
    int tile, nos;
    bool adjoint;
    int grid;
    size_t smem;
    cudaStream_t st;
    int max_smem;      // > 0: only raise the shared memory limit and report
    int *occ;          // the blocks that fit one SM
};

template <class T>
cudaError_t tile_call(const TileCall &c, const TileArgs &a, const float2 *in, float2 *out) {
    auto *kern = c.adjoint ? tile_adj_kernel<T> : tile_fwd_kernel<T>;
    if (c.max_smem > 0) {
        const cudaError_t e = raise_smem_limit(kern, c.max_smem);
        return e ? e
                 : cudaOccupancyMaxActiveBlocksPerMultiprocessor(c.occ, kern, T::THREADS, c.smem);
    }
    kern<<<c.grid, T::THREADS, c.smem, c.st>>>(a, in, out);
    return cudaGetLastError();
}

template <int W>
cudaError_t tile_width(const TileCall &c, const TileArgs &a, const float2 *in, float2 *out) {
    const bool wide = c.tile == 32;
    switch (c.nos) {
        case 32:
            return wide ? tile_call<Tile<W, 1, 32, 256>>(c, a, in, out)
                        : tile_call<Tile<W, 1, 16, 256>>(c, a, in, out);
        case 64:
            return wide ? tile_call<Tile<W, 2, 32, 256>>(c, a, in, out)
                        : tile_call<Tile<W, 2, 16, 256>>(c, a, in, out);
        case 128:
            return wide ? tile_call<Tile<W, 3, 32, 256>>(c, a, in, out)
                        : tile_call<Tile<W, 3, 16, 256>>(c, a, in, out);
        case 256: return tile_call<Tile<W, 4, 16, 256>>(c, a, in, out);
        case 512: return tile_call<Tile<W, 5, 8, 256>>(c, a, in, out);
        default: return cudaErrorInvalidValue;
    }
}

typedef cudaError_t (*TileFn)(const TileCall &, const TileArgs &, const float2 *, float2 *);

extern template cudaError_t tile_width<2>(const TileCall &, const TileArgs &, const float2 *, float2 *);
extern template cudaError_t tile_width<4>(const TileCall &, const TileArgs &, const float2 *, float2 *);
extern template cudaError_t tile_width<5>(const TileCall &, const TileArgs &, const float2 *, float2 *);
extern template cudaError_t tile_width<6>(const TileCall &, const TileArgs &, const float2 *, float2 *);
extern template cudaError_t tile_width<7>(const TileCall &, const TileArgs &, const float2 *, float2 *);
extern template cudaError_t tile_width<8>(const TileCall &, const TileArgs &, const float2 *, float2 *);
extern template cudaError_t tile_width<9>(const TileCall &, const TileArgs &, const float2 *, float2 *);
extern template cudaError_t tile_width<10>(const TileCall &, const TileArgs &, const float2 *, float2 *);
extern template cudaError_t tile_width<11>(const TileCall &, const TileArgs &, const float2 *, float2 *);
extern template cudaError_t tile_width<12>(const TileCall &, const TileArgs &, const float2 *, float2 *);

inline TileFn tile_pick(int w) {
    switch (w) {
        case 2: return tile_width<2>;
        case 4: return tile_width<4>;
        case 5: return tile_width<5>;
        case 6: return tile_width<6>;
        case 7: return tile_width<7>;
        case 8: return tile_width<8>;
        case 9: return tile_width<9>;
        case 10: return tile_width<10>;
        case 11: return tile_width<11>;
        default: return tile_width<12>;
    }
}

}  // namespace aahrt
