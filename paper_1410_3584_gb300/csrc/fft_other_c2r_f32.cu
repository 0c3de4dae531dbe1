// Complex-to-real FFT passes of the other compile-time lengths, float (see fft_other.cuh).
#include "fft_other.cuh"

namespace nlp {
template bool c2r_other<float>(float *, const DevPlan<float> &, cudaStream_t, cudaError_t &);
}  // namespace nlp
