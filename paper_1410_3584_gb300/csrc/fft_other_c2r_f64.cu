// Complex-to-real FFT passes of the other compile-time lengths, double (see fft_other.cuh).
#include "fft_other.cuh"

namespace nlp {
template bool c2r_other<double>(double *, const DevPlan<double> &, cudaStream_t, cudaError_t &);
}  // namespace nlp
