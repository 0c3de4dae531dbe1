// Real-to-complex FFT passes of the other compile-time lengths, double (see fft_other.cuh).
#include "fft_other.cuh"

namespace nlp {
template bool r2c_other<double>(const double *, const DevPlan<double> &, cudaStream_t, cudaError_t &);
}  // namespace nlp
