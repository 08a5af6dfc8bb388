// Batched fused product: several kernel settings (kernel type, bandwidth)
// over one point set share each tile's distance computation.
//
//   Y_s = (A_s + Lambda_s) V_s,  s = 0..S-1,
// A_s the kernel matrix of setting s, V_s its MS right-hand-side columns
// (typically one per regularisation value mu) and Lambda_s the per-column
// shifts.  A launch takes up to four settings of one kernel type: per pair
// (i, j) the coordinate differences of the centred points are formed once and
// give the squared l2 or the l1 distance (direct differences: no cancellation
// for clustered or duplicated points); each setting then costs one ex2 and MS
// FMAs (Matern: three more float32 operations).  The types do not share a
// launch: a difference is one of the 3 (l2) or 4 (l1) operations a coordinate
// costs, and with the type and the count known at compile time a setting has
// no branches, no unused accumulators and its scale in a register.  One kernel
// for eight settings of any types took 6.2 ms at N = 40000, d = 8, four Matern
// and four Laplace settings, two columns each (FMA pipe floor of the two
// launches: 2.5 ms, MUFU 1.7 ms); these take 3.55 ms.
// Rows are processed in packed float32x2 pairs.
#pragma once

#include "kmv_kernels.cuh"

namespace krr {

constexpr int KMVB_GROUP = 4;    // settings of one launch
constexpr int KMVB_THREADS = 256;
constexpr int KMVB_TJ = 64;

// Row pairs per thread: two while the points' coordinates leave room for both
// pairs' accumulators at two CTAs per SM, one otherwise.
__host__ __device__ constexpr int kmvb_row_pairs(int DP) { return DP <= 8 ? 2 : 1; }

struct KmvbGroup {
  int id[KMVB_GROUP];    // setting numbers: columns id MS .. id MS + MS of V and part
  float g[KMVB_GROUP];   // Gaussian: -log2e/(2 sigma^2) (times r^2)
                         // Laplace : -log2e/sigma       (times l1)
                         // Matern  : -log2e sqrt(5)/sigma (times r)
};

// xt: N x DP centred, unscaled points; V: mt x N columns; part: splits x mt x N.
template <int KERN, int DP, int CNT, int MS>
__global__ void __launch_bounds__(KMVB_THREADS, 2)
kmvb_kernel(const float *__restrict__ xt, const float *__restrict__ V, int64_t N, int mt,
            int64_t chunk, const KmvbGroup st, float *__restrict__ part) {
  constexpr int RP = kmvb_row_pairs(DP);
  constexpr int MT = CNT * MS, MTP = (MT + 1) / 2 * 2;
  constexpr int ROWS = KMVB_THREADS * 2 * RP;
  __shared__ __align__(16) float2 sx[KMVB_TJ][DP];     // {-x, -x}
  __shared__ __align__(16) float2 sv[KMVB_TJ][MTP];
  const int tid = threadIdx.x;
  const int64_t row0 = (int64_t)blockIdx.x * ROWS;
  const int64_t j_begin = (int64_t)blockIdx.y * chunk;
  const int64_t j_end = min(N, j_begin + chunk);

  float2 xi[RP][DP];
  float2 acc[RP][MT];
  float g[CNT];
#pragma unroll
  for (int s = 0; s < CNT; ++s) g[s] = st.g[s];
#pragma unroll
  for (int p = 0; p < RP; ++p) {
    const int64_t ra = row0 + tid + (int64_t)(2 * p) * KMVB_THREADS;
    const int64_t rb = ra + KMVB_THREADS;
    const bool va = ra < N, vb = rb < N;
#pragma unroll
    for (int k = 0; k < DP; ++k)
      xi[p][k] = f2(va ? xt[ra * DP + k] : 0.0f, vb ? xt[rb * DP + k] : 0.0f);
#pragma unroll
    for (int c = 0; c < MT; ++c) acc[p][c] = f2(0.0f, 0.0f);
  }

  for (int64_t j0 = j_begin; j0 < j_end; j0 += KMVB_TJ) {
    __syncthreads();
    for (int idx = tid; idx < KMVB_TJ * DP; idx += KMVB_THREADS) {
      const int64_t j = j0 + idx / DP;
      const float v = (j < j_end) ? -xt[j0 * DP + idx] : 0.0f;
      sx[idx / DP][idx % DP] = f2(v, v);
    }
#pragma unroll
    for (int c = 0; c < MTP; ++c) {
      const int64_t col = c < MT ? (int64_t)st.id[c / MS] * MS + c % MS : 0;
      for (int jj = tid; jj < KMVB_TJ; jj += KMVB_THREADS) {
        const float v = (c < MT && j0 + jj < j_end) ? V[col * N + j0 + jj] : 0.0f;
        sv[jj][c] = f2(v, v);
      }
    }
    __syncthreads();
    const int jn = (int)min((int64_t)KMVB_TJ, j_end - j0);
#pragma unroll 2
    for (int jj = 0; jj < jn; ++jj) {
      // r^2 or the l1 distance of each row pair
      float2 dist[RP];
#pragma unroll
      for (int p = 0; p < RP; ++p) dist[p] = f2(0.0f, 0.0f);
#pragma unroll
      for (int k = 0; k < DP; k += 2) {
        const float4 q = *reinterpret_cast<const float4 *>(&sx[jj][k]);
#pragma unroll
        for (int p = 0; p < RP; ++p) {
          const float2 d0 = __fadd2_rn(xi[p][k], f2(q.x, q.y));
          const float2 d1 = __fadd2_rn(xi[p][k + 1], f2(q.z, q.w));
          if constexpr (KERN == KLAPLACE) {
            dist[p].x = dist[p].x + fabsf(d0.x) + fabsf(d1.x);
            dist[p].y = dist[p].y + fabsf(d0.y) + fabsf(d1.y);
          } else {
            dist[p] = __ffma2_rn(d0, d0, dist[p]);
            dist[p] = __ffma2_rn(d1, d1, dist[p]);
          }
        }
      }
      if constexpr (KERN == KMATERN) {
#pragma unroll
        for (int p = 0; p < RP; ++p)
          dist[p] = f2(sqrt_approx(dist[p].x), sqrt_approx(dist[p].y));
      }
      float2 v[MTP];
#pragma unroll
      for (int c = 0; c < MTP; c += 2) {
        const float4 q = *reinterpret_cast<const float4 *>(&sv[jj][c]);
        v[c] = f2(q.x, q.y);
        v[c + 1] = f2(q.z, q.w);
      }
#pragma unroll
      for (int s = 0; s < CNT; ++s)
#pragma unroll
        for (int p = 0; p < RP; ++p) {
          float2 kv;
          const float2 q = __fmul2_rn(dist[p], f2(g[s], g[s]));
          if constexpr (KERN == KMATERN) {
            // q = -log2e r, r = sqrt(5) |x_i - x_j| / sigma: the exponent, and
            // 1 + r + r^2/3 in powers of q
            const float2 e = f2(ex2_approx(q.x), ex2_approx(q.y));
            const float2 poly = __ffma2_rn(
                q, __ffma2_rn(q, f2(0.16015099f, 0.16015099f), f2(-0.6931472f, -0.6931472f)),
                f2(1.0f, 1.0f));
            kv = __fmul2_rn(poly, e);
          } else {
            kv = f2(ex2_approx(q.x), ex2_approx(q.y));
          }
#pragma unroll
          for (int c = 0; c < MS; ++c)
            acc[p][s * MS + c] = __ffma2_rn(kv, v[s * MS + c], acc[p][s * MS + c]);
        }
    }
  }
  float *out = part + (int64_t)blockIdx.y * mt * N;
#pragma unroll
  for (int p = 0; p < RP; ++p) {
    const int64_t ra = row0 + tid + (int64_t)(2 * p) * KMVB_THREADS;
    const int64_t rb = ra + KMVB_THREADS;
#pragma unroll
    for (int c = 0; c < MT; ++c) {
      const int64_t col = (int64_t)st.id[c / MS] * MS + c % MS;
      if (ra < N) out[col * N + ra] = acc[p][c].x;
      if (rb < N) out[col * N + rb] = acc[p][c].y;
    }
  }
}

// Launch of one group; one translation unit per kernel type.
template <int KERN, int DP>
cudaError_t launch_kmvb_dp(int cnt, int ms, dim3 grid, cudaStream_t s, const float *xt,
                           const float *V, int64_t N, int mt, int64_t chunk, const KmvbGroup &st,
                           float *part) {
#define KRR_CASE(C, M)                                                                          \
  if (cnt == C && ms == M) {                                                                    \
    kmvb_kernel<KERN, DP, C, M><<<grid, KMVB_THREADS, 0, s>>>(xt, V, N, mt, chunk, st, part);    \
    return cudaGetLastError();                                                                  \
  }
  KRR_CASE(1, 1) KRR_CASE(2, 1) KRR_CASE(3, 1) KRR_CASE(4, 1)
  KRR_CASE(1, 2) KRR_CASE(2, 2) KRR_CASE(3, 2) KRR_CASE(4, 2)
#undef KRR_CASE
  return cudaErrorInvalidValue;
}

template <int KERN>
cudaError_t launch_kmvb(int dp, int cnt, int ms, dim3 grid, cudaStream_t s, const float *xt,
                        const float *V, int64_t N, int mt, int64_t chunk, const KmvbGroup &st,
                        float *part) {
  switch (dp) {
    case 4: return launch_kmvb_dp<KERN, 4>(cnt, ms, grid, s, xt, V, N, mt, chunk, st, part);
    case 8: return launch_kmvb_dp<KERN, 8>(cnt, ms, grid, s, xt, V, N, mt, chunk, st, part);
    case 12: return launch_kmvb_dp<KERN, 12>(cnt, ms, grid, s, xt, V, N, mt, chunk, st, part);
    case 16: return launch_kmvb_dp<KERN, 16>(cnt, ms, grid, s, xt, V, N, mt, chunk, st, part);
    case 20: return launch_kmvb_dp<KERN, 20>(cnt, ms, grid, s, xt, V, N, mt, chunk, st, part);
    case 24: return launch_kmvb_dp<KERN, 24>(cnt, ms, grid, s, xt, V, N, mt, chunk, st, part);
    case 28: return launch_kmvb_dp<KERN, 28>(cnt, ms, grid, s, xt, V, N, mt, chunk, st, part);
    case 32: return launch_kmvb_dp<KERN, 32>(cnt, ms, grid, s, xt, V, N, mt, chunk, st, part);
  }
  return cudaErrorInvalidValue;
}

}  // namespace krr
