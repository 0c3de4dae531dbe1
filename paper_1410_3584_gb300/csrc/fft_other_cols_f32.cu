// Column FFT passes of the other compile-time lengths, float (see fft_other.cuh).
#include "fft_other.cuh"

namespace nlp {
template bool cols_other<float>(cpx<float> *, const StridedDesc &, const FftLen<float> &, int, cudaStream_t, cudaError_t &);
}  // namespace nlp
