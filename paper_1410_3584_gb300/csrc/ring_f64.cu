// Ring kernels, double instantiations (see ring_launch.cuh).
#include <algorithm>
#include <type_traits>

#include "ring_launch.cuh"

namespace nlp {
template size_t ring_smem<double>(const DevPlan<double> &, int);
template int ring_psi_stride<double>(int);
template cudaError_t launch_ring_cols<double>(const DevPlan<double> &, cudaStream_t);
template cudaError_t launch_ring_nodes<double>(const DevPlan<double> &, cudaStream_t);
template cudaError_t launch_ring_inv<double>(const DevPlan<double> &, cudaStream_t);
template cudaError_t launch_ring_gather<double>(const DevPlan<double> &, cudaStream_t);
template cudaError_t launch_ring_gather2<double>(const DevPlan<double> &, cudaStream_t);
template int ring_xy_stride<double>(int);
}  // namespace nlp
