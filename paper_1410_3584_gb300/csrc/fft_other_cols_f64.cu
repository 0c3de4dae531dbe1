// Column FFT passes of the other compile-time lengths, double (see fft_other.cuh).
#include "fft_other.cuh"

namespace nlp {
template bool cols_other<double>(cpx<double> *, const StridedDesc &, const FftLen<double> &, int, cudaStream_t, cudaError_t &);
}  // namespace nlp
