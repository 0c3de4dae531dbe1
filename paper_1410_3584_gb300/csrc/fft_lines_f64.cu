// Four-step column passes and contiguous complex FFT passes, double (see fft_launch.cuh).
#include "fft_launch.cuh"

namespace nlp {
template cudaError_t launch_fft_four<double>(const cpx<double> *, cpx<double> *, const StridedDesc &, const DevPlan<double> &, int,
                                         cudaStream_t);
template cudaError_t launch_fft_contig<double>(cpx<double> *, int64_t, const FftLen<double> &, int, double, cudaStream_t);
}  // namespace nlp
