// Instantiates the fixed-point float-float products for one kernel function.
#include "kmvfix_kernels.cuh"

namespace krr {

cudaError_t launch_kmvfix_ff_gauss(int DP, int M, dim3 grid, cudaStream_t s, const KmvFixArgs &a) {
  return launch_kmvfix<FixAccFF, KGAUSS>(DP, M, grid, s, a);
}

}  // namespace krr
