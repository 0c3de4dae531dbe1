// Ring kernels, float instantiations (see ring_launch.cuh).
#include <algorithm>
#include <type_traits>

#include "ring_launch.cuh"

namespace nlp {
template size_t ring_smem<float>(const DevPlan<float> &, int);
template int ring_psi_stride<float>(int);
template cudaError_t launch_ring_cols<float>(const DevPlan<float> &, cudaStream_t);
template cudaError_t launch_ring_nodes<float>(const DevPlan<float> &, cudaStream_t);
template cudaError_t launch_ring_inv<float>(const DevPlan<float> &, cudaStream_t);
template cudaError_t launch_ring_gather<float>(const DevPlan<float> &, cudaStream_t);
template cudaError_t launch_ring_gather2<float>(const DevPlan<float> &, cudaStream_t);
template int ring_xy_stride<float>(int);
}  // namespace nlp
