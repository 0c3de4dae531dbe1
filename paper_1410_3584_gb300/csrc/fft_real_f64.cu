// Last-axis FFT passes (real to complex, complex to real), double (see fft_launch.cuh).
#include "fft_launch.cuh"

namespace nlp {
template cudaError_t launch_fwd_r2c<double>(const double *, const DevPlan<double> &, cudaStream_t);
template cudaError_t launch_inv_c2r<double>(double *, const DevPlan<double> &, cudaStream_t);
}  // namespace nlp
