// Instantiates the fixed-point float64 products and columns for one kernel function.
#include "kmvfix_kernels.cuh"

namespace krr {

cudaError_t launch_kmvfix_laplace(int DP, int M, dim3 grid, cudaStream_t s, const KmvFixArgs &a) {
  return launch_kmvfix<FixAccD, KLAPLACE>(DP, M, grid, s, a);
}

cudaError_t launch_kfix_columns_laplace(int DP, const int2 *ua, int64_t N, const FixScale *scale,
                                   const int64_t *cols, int nc, double *G, int64_t ldg,
                                   cudaStream_t s) {
  return launch_kfix_columns<KLAPLACE>(DP, ua, N, scale, cols, nc, G, ldg, s);
}

}  // namespace krr
