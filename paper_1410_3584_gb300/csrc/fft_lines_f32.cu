// Four-step column passes and contiguous complex FFT passes, float (see fft_launch.cuh).
#include "fft_launch.cuh"

namespace nlp {
template cudaError_t launch_fft_four<float>(const cpx<float> *, cpx<float> *, const StridedDesc &, const DevPlan<float> &, int,
                                         cudaStream_t);
template cudaError_t launch_fft_contig<float>(cpx<float> *, int64_t, const FftLen<float> &, int, float, cudaStream_t);
}  // namespace nlp
