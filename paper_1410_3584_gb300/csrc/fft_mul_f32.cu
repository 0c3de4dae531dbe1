// Column passes fused with a pointwise product, float (see fft_launch.cuh).
#include "fft_launch.cuh"

namespace nlp {
template cudaError_t launch_fft_mul<float, float>(cpx<float> *, const StridedDesc &, const FftLen<float> &,
                                                    const float *, cudaStream_t);
template cudaError_t launch_fft_mul<float, cpx<float>>(cpx<float> *, const StridedDesc &, const FftLen<float> &,
                                                         const cpx<float> *, cudaStream_t);
template cudaError_t launch_fft_mul3<float>(cpx<float> *, const StridedDesc &, const FftLen<float> &,
                                            const cpx<double> *, const cpx<double> *, const cpx<double> *, cudaStream_t);
}  // namespace nlp
