// Column passes fused with a pointwise product, double (see fft_launch.cuh).
#include "fft_launch.cuh"

namespace nlp {
bool fft_fixed_len(int N) {
    FftLen<double> L{};
    L.N = N;
    return with_fixed_len(L, [](auto) {});
}
template cudaError_t launch_fft_mul<double, double>(cpx<double> *, const StridedDesc &, const FftLen<double> &,
                                                    const double *, cudaStream_t);
template cudaError_t launch_fft_mul<double, cpx<double>>(cpx<double> *, const StridedDesc &, const FftLen<double> &,
                                                         const cpx<double> *, cudaStream_t);
template cudaError_t launch_fft_mul3<double>(cpx<double> *, const StridedDesc &, const FftLen<double> &,
                                            const cpx<double> *, const cpx<double> *, const cpx<double> *, cudaStream_t);
}  // namespace nlp
