// Register-FFT time kernels of 2048-sample frames.
#include "time_fft_dispatch.cuh"

namespace aahrt {

template cudaError_t frame_call<8>(const FrameCall &, const FrameArgs &, const void *, void *, const float *);

}  // namespace aahrt
