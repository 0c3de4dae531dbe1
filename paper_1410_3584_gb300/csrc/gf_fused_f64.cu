// Fused gradient-flow passes, double (see gf_fused.cuh).
#include "gf_fused.cuh"

namespace nlp {
template cudaError_t launch_gf_r2c<double>(const double *, const double *, const double *, double, const double *, const int *,
                                           const DevPlan<double> &, cudaStream_t);
template cudaError_t launch_gf_c2r<double>(double *, double *, const DevPlan<double> &, double *, int *, int, double, cudaStream_t);
}  // namespace nlp
