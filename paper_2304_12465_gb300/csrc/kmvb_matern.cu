// Instantiates the batched product for one kernel function.
#include "kmvb_kernels.cuh"

namespace krr {

cudaError_t launch_kmvb_matern(int dp, int cnt, int ms, dim3 grid, cudaStream_t s, const float *xt,
                           const float *V, int64_t N, int mt, int64_t chunk, const KmvbGroup &st,
                           float *part) {
  return launch_kmvb<KMATERN>(dp, cnt, ms, grid, s, xt, V, N, mt, chunk, st, part);
}

}  // namespace krr
