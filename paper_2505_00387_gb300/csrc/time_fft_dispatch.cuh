// The register-FFT time kernels of one frame length (time_fft.cuh) behind one
// function, compiled in separate files so they build in parallel.
#pragma once

#include "time_fft.cuh"

namespace aahrt {

// (GATHER_*: gathers fastest)
enum FrameOp { FRAME_R2C, FRAME_C2R, FRAME_FUSED, GATHER_R2C, GATHER_C2R };

struct FrameCall {
    FrameOp op;
    bool model_side;     // columns of the model (S, S^T), else of the data (U, U^T)
    int interp, epi, pairs;
    cudaStream_t st;
    int max_smem;        // > 0: only raise the kernels' shared memory limit
};

template <class F, class K, class... A>
cudaError_t frame_run(const FrameCall &c, const FrameArgs &a, int nrows, K *kern, A... args) {
    if (c.max_smem > 0) return raise_smem_limit(kern, c.max_smem);
    const int per = c.pairs * a.seq;       // pairs a block owns
    const int grid = (a.ngroups + per - 1) / per;
    kern<<<grid, F::T * c.pairs, frame_smem<F>(c.pairs, a.seq, nrows, a.nfrac), c.st>>>(a, args...);
    return cudaGetLastError();
}

template <class F, int INTERP>
cudaError_t frame_interp(const FrameCall &c, const FrameArgs &a, const void *in, void *out,
                         const float *aux) {
    const float *fi = static_cast<const float *>(in);
    const float2 *ci = static_cast<const float2 *>(in);
    float *fo = static_cast<float *>(out);
    float2 *co = static_cast<float2 *>(out);
    if (c.op >= GATHER_R2C) {
        if (c.op == GATHER_R2C)
            return c.model_side
                       ? frame_run<F>(c, a, a.nrows, gather_r2c_kernel<F, INTERP, false>, fi, co)
                       : frame_run<F>(c, a, a.nrows, gather_r2c_kernel<F, INTERP, true>, fi, co);
        if (c.model_side)
            return frame_run<F>(c, a, 0, gather_c2r_kernel<F, INTERP, true, EPI_STORE>, ci, fo, aux);
        return c.epi == EPI_RESIDUAL
                   ? frame_run<F>(c, a, 0, gather_c2r_kernel<F, INTERP, false, EPI_RESIDUAL>, ci, fo,
                                  aux)
                   : frame_run<F>(c, a, 0, gather_c2r_kernel<F, INTERP, false, EPI_STORE>, ci, fo,
                                  aux);
    }
    if (c.op == FRAME_R2C)
        return c.model_side
                   ? frame_run<F>(c, a, a.nrows, frame_r2c_kernel<F, INTERP, false>, fi, co)
                   : frame_run<F>(c, a, a.nrows, frame_r2c_kernel<F, INTERP, true>, fi, co);
    if (c.op == FRAME_FUSED)
        return c.model_side
                   ? frame_run<F>(c, a, a.nrows, frame_fused_kernel<F, INTERP, true, EPI_FISTA>, co,
                                  aux)
                   : frame_run<F>(c, a, a.nrows, frame_fused_kernel<F, INTERP, false, EPI_RESIDUAL>,
                                  co, aux);
    if (c.model_side)
        return c.epi == EPI_FISTA
                   ? frame_run<F>(c, a, 0, frame_c2r_kernel<F, INTERP, true, EPI_FISTA>, ci, fo, aux)
                   : frame_run<F>(c, a, 0, frame_c2r_kernel<F, INTERP, true, EPI_STORE>, ci, fo, aux);
    return c.epi == EPI_RESIDUAL
               ? frame_run<F>(c, a, 0, frame_c2r_kernel<F, INTERP, false, EPI_RESIDUAL>, ci, fo, aux)
               : frame_run<F>(c, a, 0, frame_c2r_kernel<F, INTERP, false, EPI_STORE>, ci, fo, aux);
}

template <int C>
cudaError_t frame_call(const FrameCall &c, const FrameArgs &a, const void *in, void *out,
                       const float *aux) {
    return c.interp == AAHRT_INTERP_LINEAR
               ? frame_interp<Frame<C>, AAHRT_INTERP_LINEAR>(c, a, in, out, aux)
               : frame_interp<Frame<C>, AAHRT_INTERP_KEYS>(c, a, in, out, aux);
}

typedef cudaError_t (*FrameFn)(const FrameCall &, const FrameArgs &, const void *, void *,
                               const float *);

extern template cudaError_t frame_call<2>(const FrameCall &, const FrameArgs &, const void *, void *, const float *);
extern template cudaError_t frame_call<4>(const FrameCall &, const FrameArgs &, const void *, void *, const float *);
extern template cudaError_t frame_call<8>(const FrameCall &, const FrameArgs &, const void *, void *, const float *);
extern template cudaError_t frame_call<16>(const FrameCall &, const FrameArgs &, const void *, void *, const float *);
extern template cudaError_t frame_call<32>(const FrameCall &, const FrameArgs &, const void *, void *, const float *);

}  // namespace aahrt
