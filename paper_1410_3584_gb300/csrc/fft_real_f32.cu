// Last-axis FFT passes (real to complex, complex to real), float (see fft_launch.cuh).
#include "fft_launch.cuh"

namespace nlp {
template cudaError_t launch_fwd_r2c<float>(const float *, const DevPlan<float> &, cudaStream_t);
template cudaError_t launch_inv_c2r<float>(float *, const DevPlan<float> &, cudaStream_t);
}  // namespace nlp
