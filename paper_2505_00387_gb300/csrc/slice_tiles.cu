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

// One cube's block of [rows][cols] -> [cols][rows], in tiles of 32 x 64 (64 x 64:
// 4 % more of a stage).  BOUND (rows = bins): also the largest |re| + |im| of
// each chunk of bins (of 64 or more, so a tile lies in one) into the cube's row
// of the bound table, where a pass of its own over the spectrum per azimuth
// group took a third of stage 4.
constexpr int kRows = 32;
template <bool BOUND>
__global__ void __launch_bounds__(256)
transpose_kernel(const float2 *__restrict__ in, float2 *__restrict__ out,
                 const SpecBlock *__restrict__ blk, int nbins, int to_bins, unsigned *ymax,
                 int nychunk, int ychunk_log) {
    __shared__ float2 s[kRows][65];
    __shared__ unsigned s_max;
    const SpecBlock b = blk[blockIdx.z];
    const int rows = to_bins ? nbins : b.ncol, cols = to_bins ? b.ncol : nbins;
    const int tx = threadIdx.x & 63, ty = threadIdx.x >> 6;
    const int ox = threadIdx.x % kRows, oy = threadIdx.x / kRows;
    const int c0 = blockIdx.x * 64;
    if (c0 >= cols) return;              // (a cube of fewer columns than the largest)
    for (int r0 = blockIdx.y * kRows; r0 < rows; r0 += gridDim.y * kRows) {
        float2 v[kRows / 4];
#pragma unroll
        for (int i = 0; i < kRows / 4; ++i) {
            v[i] = make_float2(0.f, 0.f);
            if (r0 + ty + 4 * i < rows && c0 + tx < cols)
                v[i] = __ldcs(in + b.off + (long long)(r0 + ty + 4 * i) * cols + c0 + tx);
        }
        if (BOUND && threadIdx.x == 0) s_max = 0u;
        float m = 0.f;
#pragma unroll
        for (int i = 0; i < kRows / 4; ++i) {
            s[ty + 4 * i][tx] = v[i];
            m = fmaxf(m, fabsf(v[i].x) + fabsf(v[i].y));
        }
        __syncthreads();
        if (BOUND) {
            const unsigned w = __reduce_max_sync(0xffffffffu, __float_as_uint(m));
            if ((threadIdx.x & 31) == 0 && w > 0u) atomicMax(&s_max, w);
        }
#pragma unroll
        for (int i = 0; i < kRows / 4; ++i) {
            const int c = oy + i * (256 / kRows);
            if (c0 + c < cols && r0 + ox < rows)
                out[b.off + (long long)(c0 + c) * rows + r0 + ox] = s[ox][c];
        }
        __syncthreads();
        if (BOUND && threadIdx.x == 0) {
            unsigned *e = ymax + (long long)blockIdx.z * nychunk + (r0 >> ychunk_log);
            if (s_max > *(volatile unsigned *)e) atomicMax(e, s_max);
        }
    }
}

cudaError_t launch_transpose_spec(Plan &p, bool model_side, const float2 *in, float2 *out,
                                  bool to_bins, bool bound, cudaStream_t st) {
    cudaError_t e;
    if (bound && (e = ybound_begin(p, st))) return e;
    const SpecBlock *blk = model_side ? p.spec_model : p.spec_data;
    const int ncol = model_side ? (int)p.cols_model : p.max_ntr;
    const int rows = to_bins ? p.nbins : ncol, cols = to_bins ? ncol : p.nbins;
    auto *kern = bound ? transpose_kernel<true> : transpose_kernel<false>;
    for (int c0 = 0; c0 < p.ncube; c0 += 65535)
        kern<<<dim3((cols + 63) / 64, std::min((rows + kRows - 1) / kRows, 65535),
                    std::min(p.ncube - c0, 65535)), 256, 0, st>>>(
            in, out, blk + c0, p.nbins, to_bins ? 1 : 0, p.ymax + (long long)c0 * p.nychunk,
            p.nychunk, p.ychunk_log);
    p.launches[6]++;
    return cudaGetLastError();
}

}  // namespace aahrt
