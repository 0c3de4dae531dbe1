// Real-to-complex FFT passes of the other compile-time lengths, float (see fft_other.cuh).
#include "fft_other.cuh"

namespace nlp {
template bool r2c_other<float>(const float *, const DevPlan<float> &, cudaStream_t, cudaError_t &);
}  // namespace nlp
