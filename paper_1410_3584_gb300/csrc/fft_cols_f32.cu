// Column FFT passes, float (see fft_launch.cuh).
#include "fft_launch.cuh"

namespace nlp {
template cudaError_t launch_fft_strided<float>(cpx<float> *, const StridedDesc &, const FftLen<float> &, int, cudaStream_t);
template bool cols_on_reg_engine<float>(const FftLen<float> &);
}  // namespace nlp
