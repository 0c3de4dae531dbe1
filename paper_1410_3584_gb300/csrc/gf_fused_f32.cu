// Fused gradient-flow passes, float (see gf_fused.cuh).
#include "gf_fused.cuh"

namespace nlp {
template cudaError_t launch_gf_r2c<float>(const float *, const float *, const float *, float, const double *, const int *,
                                           const DevPlan<float> &, cudaStream_t);
template cudaError_t launch_gf_c2r<float>(float *, float *, const DevPlan<float> &, double *, int *, int, double, cudaStream_t);
}  // namespace nlp
