// Dispatch of the bins-fastest slice kernels (slice_tiles.cuh) and the
// transposition between the two spectrum layouts.
#include <algorithm>

#include "slice_tiles_dispatch.cuh"

namespace aahrt {

static TileArgs tile_args(const Plan &p, int *counter) {
    TileArgs a;
    a.geo = p.geo;
    a.groups = p.groups;
    a.slice_start = p.slice_start;
    a.dec = p.dec;
    a.tw = p.tw_q;
    a.counter = counter;
    a.nbins = p.nbins;
    a.ntiles = (p.nbins + p.tile - 1) / p.tile;
    a.total = (long long)p.ngroups_total * a.ntiles;
    a.nq = p.nq;
    a.ntheta = p.ntheta;
    a.nos = p.nos;
    a.Lq = p.Lq;
    a.cq = p.cq;
    a.scale = (float)(1.0 / p.nfft);
    a.phicap = (float)p.phicap;
    a.ymax = p.ymax;
    a.wsum = p.wsum;
    a.ncube = p.ncube;
    a.nychunk = p.nychunk;
    a.ychunk_log = p.ychunk_log;
    a.poly = p.poly;
    return a;
}

cudaError_t launch_slice_tiles(Plan &p, bool adjoint, const float2 *in, float2 *out,
                               cudaStream_t st, int *counter) {
    const TileArgs a = tile_args(p, counter);
    const int grid = adjoint ? p.slice_grid_adj : p.slice_grid_fwd;
    const size_t smem = adjoint ? p.smem_sadj : p.smem_sfwd;
    return tile_pick(p.w)(TileCall{p.tile, p.nos, adjoint, grid, smem, st, 0, nullptr}, a, in, out);
}

cudaError_t configure_tile_kernels(Plan &p, int num_sms, int max_smem) {
    p.smem_sfwd = p.smem_sadj = tile_smem(p.nos, p.w, p.tile);
    const long long items = (long long)p.ngroups_total * ((p.nbins + p.tile - 1) / p.tile);
    for (int adj = 0; adj < 2; ++adj) {
        int occ = 0;
        const TileArgs none{};
        cudaError_t e = tile_pick(p.w)(
            TileCall{p.tile, p.nos, adj != 0, 0, p.smem_sfwd, nullptr, max_smem, &occ}, none,
            nullptr, nullptr);
        if (e) return e;
        if (occ < 1) return cudaErrorInvalidConfiguration;
        (adj ? p.slice_grid_adj : p.slice_grid_fwd) =
            (int)std::min<long long>(items, (long long)occ * num_sms);
    }
    return cudaSuccess;
}

// One cube's block of [rows][cols] -> [cols][rows], 32 x 32 tiles.
__global__ void transpose_kernel(const float2 *__restrict__ in, float2 *__restrict__ out,
                                 const SpecBlock *__restrict__ blk, int nbins, int to_bins) {
    __shared__ float2 s[32][33];
    const SpecBlock b = blk[blockIdx.z];
    const int rows = to_bins ? nbins : b.ncol, cols = to_bins ? b.ncol : nbins;
    const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
    for (int r0 = blockIdx.y * 32; r0 < rows; r0 += gridDim.y * 32)
        for (int c0 = blockIdx.x * 32; c0 < cols; c0 += gridDim.x * 32) {
            for (int i = ty; i < 32; i += 8)
                if (r0 + i < rows && c0 + tx < cols)
                    s[i][tx] = in[b.off + (long long)(r0 + i) * cols + c0 + tx];
            __syncthreads();
            for (int i = ty; i < 32; i += 8)
                if (c0 + i < cols && r0 + tx < rows)
                    out[b.off + (long long)(c0 + i) * rows + r0 + tx] = s[tx][i];
            __syncthreads();
        }
}

cudaError_t launch_transpose_spec(Plan &p, bool model_side, const float2 *in, float2 *out,
                                  bool to_bins, cudaStream_t st) {
    const SpecBlock *blk = model_side ? p.spec_model : p.spec_data;
    const int ncol = model_side ? (int)p.cols_model : p.max_ntr;
    const int gr = ((to_bins ? p.nbins : ncol) + 31) / 32, gc = ((to_bins ? ncol : p.nbins) + 31) / 32;
    for (int c0 = 0; c0 < p.ncube; c0 += 65535) {
        const int n = std::min(p.ncube - c0, 65535);
        transpose_kernel<<<dim3(gc, std::min(gr, 65535), n), 256, 0, st>>>(in, out, blk + c0, p.nbins,
                                                                          to_bins ? 1 : 0);
    }
    return cudaGetLastError();
}

}  // namespace aahrt
