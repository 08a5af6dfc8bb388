// Instantiates the symmetric fixed-point products for one kernel function.
#include "kmvfix_kernels.cuh"

namespace krr {

cudaError_t launch_kmvfixsym_gauss(int DP, int M, cudaStream_t s, const KmvFixSymArgs &a) {
  return launch_kmvfixsym<FixAccD, KGAUSS>(DP, M, s, a);
}

}  // namespace krr
