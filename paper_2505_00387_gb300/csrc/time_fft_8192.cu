// Register-FFT time kernels of 8192-sample frames.
#include "time_fft_dispatch.cuh"

namespace aahrt {

template cudaError_t frame_call<32>(const FrameCall &, const FrameArgs &, const void *, void *, const float *);

}  // namespace aahrt
