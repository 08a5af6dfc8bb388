// Host driver of the batched multi-setting fused product (kmvb_kernels.cuh).
#include <algorithm>
#include <cmath>

#include "kmv.cuh"
#include "kmvb_kernels.cuh"

namespace krr {

#define KRR_DECL(K)                                                                          \
  cudaError_t launch_kmvb_##K(int dp, int cnt, int ms, dim3 grid, cudaStream_t s,              \
                              const float *xt, const float *V, int64_t N, int mt,             \
                              int64_t chunk, const KmvbGroup &st, float *part);
KRR_DECL(gauss)
KRR_DECL(laplace)
KRR_DECL(matern)
#undef KRR_DECL

// Y[c] = lambda[c] V[c] + the splits' sums: 32 rows a block, whose eight warps
// take every eighth split each.
constexpr int KMVB_RED_WARPS = 8;
__global__ void __launch_bounds__(32 * KMVB_RED_WARPS)
kmvb_reduce_kernel(const float *__restrict__ part, int splits, int64_t N, int mt,
                   const float *__restrict__ lambda, const float *__restrict__ V,
                   float *__restrict__ Y) {
  __shared__ float red[KMVB_RED_WARPS][32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, c = blockIdx.y;
  const int64_t i = (int64_t)blockIdx.x * 32 + lane;
  float acc = 0.0f;
  if (i < N) {
#pragma unroll 4
    for (int sp = warp; sp < splits; sp += KMVB_RED_WARPS)
      acc += part[((int64_t)sp * mt + c) * N + i];
  }
  red[warp][lane] = acc;
  __syncthreads();
  if (warp != 0 || i >= N) return;
#pragma unroll
  for (int w = 1; w < KMVB_RED_WARPS; ++w) acc += red[w][lane];
  Y[(int64_t)c * N + i] = acc + lambda[c] * V[(int64_t)c * N + i];
}

krr_status kmvb_prepare(const double *Xd, int64_t N, int d, cudaStream_t s, PointsF32 &P) {
  // centred, unscaled points: every setting applies its own scale
  return prepare_points_f32(Xd, N, d, KLAPLACE, 1.4426950408889634, s, P);
}

krr_status kmv_batched_f32(const PointsF32 &P, int S, const int *kerns, const double *sigmas,
                           int ms, const float *lambda_dev, const float *V, float *Y,
                           cudaStream_t s, DevBuf<float> &part) {
  const int64_t N = P.N;
  if (N == 0 || S == 0) return KRR_OK;
  // groups of up to KMVB_GROUP settings of one type
  const int mt = S * ms;
  const double log2e = 1.4426950408889634;
  const int rows = KMVB_THREADS * 2 * kmvb_row_pairs(P.dp);
  const int64_t row_tiles = (N + rows - 1) / rows;
  // about eight waves of two CTAs a SM: short enough float32 sums, and a last
  // wave that costs little
  int64_t splits = ((int64_t)num_sms() * 2 * 8 + row_tiles - 1) / row_tiles;
  splits = std::min(splits, (N + KMVB_TJ - 1) / KMVB_TJ);
  int64_t chunk = (N + splits - 1) / splits;
  chunk = (chunk + KMVB_TJ - 1) / KMVB_TJ * KMVB_TJ;
  const int nsplit = (int)((N + chunk - 1) / chunk);
  const size_t need = (size_t)nsplit * mt * N;
  if (part.n < need) KRR_TRY(part.alloc(need, s));
  const dim3 grid((unsigned)row_tiles, nsplit);
  for (int type : {KGAUSS, KLAPLACE, KMATERN}) {
    KmvbGroup st{};
    int cnt = 0;
    for (int q = 0; q <= S; ++q) {
      if (q < S && kerns[q] == type) {
        const double sg = sigmas[q];
        st.id[cnt] = q;
        st.g[cnt++] = (float)(type == KGAUSS     ? -log2e / (2.0 * sg * sg)
                              : type == KLAPLACE ? -log2e / sg
                                                 : -log2e * std::sqrt(5.0) / sg);
      }
      if (cnt == 0 || (q < S && cnt < KMVB_GROUP)) continue;
      const auto launch = type == KGAUSS ? launch_kmvb_gauss
                          : type == KLAPLACE ? launch_kmvb_laplace : launch_kmvb_matern;
      const cudaError_t e = launch(P.dp, cnt, ms, grid, s, P.xt.p, V, N, mt, chunk, st, part.p);
      count_launch();
      if (e != cudaSuccess) {
        set_error("batched product launch failed: %s", cudaGetErrorString(e));
        return KRR_ECUDA;
      }
      cnt = 0;
    }
  }
  kmvb_reduce_kernel<<<dim3(ceil_div(N, 32), mt), 32 * KMVB_RED_WARPS, 0, s>>>(
      part.p, nsplit, N, mt, lambda_dev, V, Y);
  KRR_LAUNCH_CHECK();
  return KRR_OK;
}

}  // namespace krr
