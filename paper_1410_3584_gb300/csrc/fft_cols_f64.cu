// Column FFT passes, double (see fft_launch.cuh).
#include "fft_launch.cuh"

namespace nlp {
template cudaError_t launch_fft_strided<double>(cpx<double> *, const StridedDesc &, const FftLen<double> &, int, cudaStream_t);
template bool cols_on_reg_engine<double>(const FftLen<double> &);
}  // namespace nlp
