// Instantiates the two-pass kernels for the register report.
#include "lbm_kernels_split.cuh"

namespace lbm {
template __global__ void split_moments_kernel<float>(LatticeDesc);
template __global__ void split_moments_kernel<double>(LatticeDesc);
#define LBM_SPLIT(T, ST)                                              \
  template __global__ void split_collide_kernel<T, ST, true>(LatticeDesc); \
  template __global__ void split_collide_kernel<T, ST, false>(LatticeDesc);
LBM_SPLIT(float, 4)
LBM_SPLIT(float, 6)
LBM_SPLIT(float, 8)
LBM_SPLIT(double, 4)
LBM_SPLIT(double, 6)
LBM_SPLIT(double, 8)
}  // namespace lbm
