// Float64 products and kernel columns on fixed-point kernel values (kfix.cuh).
//
// The integer pipe bounds them: per entry 3d multiply-adds for the sums of
// squares plus about 15 for 2^-E, at 53 a clock and SM, then one DFMA per
// right-hand side (1.9 a clock and SM).  A thread keeps two rows' limbs in
// registers (one for d > 16, where two would spill) and walks a shared tile
// of columns, which every lane reads at the same address.  Measured, Gaussian,
// N = 4096, d = 8, one right-hand side: 110 us (2.06 clocks an entry and SM)
// against 1055 us for kmv64_kernel; 20 kernel columns there 7.3 us against
// 34.7.
#pragma once

#include "kfix.cuh"
#include "kmv.cuh"

namespace krr {

constexpr int KFIX_THREADS = 128;
constexpr int KFIX_TJ = 32;

__host__ __device__ constexpr int kmvfix_rows_per_thread(int DP) { return DP <= 16 ? 2 : 1; }

// kappa of one pair from the row's coordinates (registers) and the column's
// (shared, 16-byte aligned).
template <int KERN, int DP>
__device__ __forceinline__ double fix_kappa(const int2 (&u)[DP], const int4 *__restrict__ v,
                                            const FixScale &fs,
                                            const uint64_t *__restrict__ tab) {
  if constexpr (KERN == KLAPLACE) {
    uint64_t S = 0;
#pragma unroll
    for (int k = 0; k < DP; k += 2) {
      const int4 b = v[k / 2];
      const int64_t d0 = (int64_t)(((uint64_t)(uint32_t)u[k].y << 32) | (uint32_t)u[k].x) -
                         (int64_t)(((uint64_t)(uint32_t)b.y << 32) | (uint32_t)b.x);
      const int64_t d1 = (int64_t)(((uint64_t)(uint32_t)u[k + 1].y << 32) | (uint32_t)u[k + 1].x) -
                         (int64_t)(((uint64_t)(uint32_t)b.w << 32) | (uint32_t)b.z);
      S += (uint64_t)llabs(d0) + (uint64_t)llabs(d1);
    }
    return fix_exp2(fix_exponent_l1(S, fs.r), tab);
  } else {
    int64_t S1 = 0, S2 = 0;
    uint64_t S3 = 0;
#pragma unroll
    for (int k = 0; k < DP; k += 2) {
      const int4 b = v[k / 2];
      const int h0 = u[k].x - b.x, l0 = u[k].y - b.y;
      const int h1 = u[k + 1].x - b.z, l1 = u[k + 1].y - b.w;
      S1 += (int64_t)h0 * h0;
      S2 += (int64_t)h0 * l0;
      S3 += (uint64_t)((int64_t)l0 * l0);
      S1 += (int64_t)h1 * h1;
      S2 += (int64_t)h1 * l1;
      S3 += (uint64_t)((int64_t)l1 * l1);
    }
    if constexpr (KERN == KMATERN) return fix_matern(S1, S2, S3, fs.r2_scale, tab);
    else return fix_exp2(fix_exponent(S1, S2, S3, fs.r, fs.s1_max), tab);
  }
}

// part[split][c][row] = sum over the split's columns of kappa v; ur (Nr x DP),
// uc (N x DP): coordinates of rows and columns.
template <int KERN, int DP, int M>
__global__ void __launch_bounds__(KFIX_THREADS)
kmvfix_kernel(const int2 *__restrict__ ur, int64_t Nr, const int2 *__restrict__ uc,
              const FixScale *__restrict__ scale, const double *__restrict__ V, int64_t ldv,
              int64_t N, int m, int64_t chunk, double *__restrict__ part) {
  constexpr int RI = kmvfix_rows_per_thread(DP);
  __shared__ __align__(16) int2 su[KFIX_TJ][DP];
  __shared__ double sv[KFIX_TJ][M];
  __shared__ uint64_t tab[kFixTab];
  if (!scale->ok) return;
  const int tid = threadIdx.x;
  FixScale fs;
  fs.r = scale->r;
  fs.s1_max = scale->s1_max;
  fs.r2_scale = scale->r2_scale;
  for (int i = tid; i < kFixTab; i += KFIX_THREADS) tab[i] = kFixExp2Tab[i];
  const int64_t row0 = (int64_t)blockIdx.x * (KFIX_THREADS * RI) + tid;
  const int64_t j_begin = (int64_t)blockIdx.y * chunk;
  const int64_t j_end = min(N, j_begin + chunk);
  int2 u[RI][DP];
  double acc[RI][M];
#pragma unroll
  for (int r = 0; r < RI; ++r) {
    const int64_t i = min(row0 + (int64_t)r * KFIX_THREADS, Nr - 1);
    const int4 *src = reinterpret_cast<const int4 *>(ur + i * DP);
#pragma unroll
    for (int k = 0; k < DP; k += 2) {
      const int4 q = src[k / 2];
      u[r][k] = make_int2(q.x, q.y);
      u[r][k + 1] = make_int2(q.z, q.w);
    }
#pragma unroll
    for (int c = 0; c < M; ++c) acc[r][c] = 0.0;
  }
  for (int64_t j0 = j_begin; j0 < j_end; j0 += KFIX_TJ) {
    const int jn = (int)min((int64_t)KFIX_TJ, j_end - j0);
    __syncthreads();
    const int4 *src = reinterpret_cast<const int4 *>(uc + j0 * DP);
    for (int i = tid; i < jn * (DP / 2); i += KFIX_THREADS)
      reinterpret_cast<int4 *>(su)[i] = src[i];
    for (int i = tid; i < KFIX_TJ * M; i += KFIX_THREADS) {
      const int c = i / KFIX_TJ, jj = i % KFIX_TJ;
      sv[jj][c] = (jj < jn && c < m) ? V[(int64_t)c * ldv + j0 + jj] : 0.0;
    }
    __syncthreads();
#pragma unroll 1
    for (int jj = 0; jj < jn; ++jj) {
      const int4 *v = reinterpret_cast<const int4 *>(su[jj]);
      double kv[RI];
#pragma unroll
      for (int r = 0; r < RI; ++r) kv[r] = fix_kappa<KERN, DP>(u[r], v, fs, tab);
#pragma unroll
      for (int c = 0; c < M; ++c)
#pragma unroll
        for (int r = 0; r < RI; ++r) acc[r][c] = fma(kv[r], sv[jj][c], acc[r][c]);
    }
  }
  double *out = part + (int64_t)blockIdx.y * M * Nr;
#pragma unroll
  for (int r = 0; r < RI; ++r) {
    const int64_t i = row0 + (int64_t)r * KFIX_THREADS;
    if (i < Nr)
#pragma unroll
      for (int c = 0; c < M; ++c)
        if (c < m) out[(int64_t)c * Nr + i] = acc[r][c];
  }
}

// G(i, c) = kappa(x_i, x_cols[c]) for all rows i and nc
// columns (ld ldg, column-major); ua: N x DP.
template <int KERN, int DP>
__global__ void __launch_bounds__(KFIX_THREADS)
kfix_columns_kernel(const int2 *__restrict__ ua, int64_t N, const FixScale *__restrict__ scale,
                    const int64_t *__restrict__ cols, int nc, double *__restrict__ G,
                    int64_t ldg) {
  constexpr int COLS = 32;   // columns per CTA (blockIdx.y picks the group)
  __shared__ __align__(16) int2 su[COLS][DP];
  __shared__ uint64_t tab[kFixTab];
  if (!scale->ok) return;
  const int tid = threadIdx.x;
  FixScale fs;
  fs.r = scale->r;
  fs.s1_max = scale->s1_max;
  fs.r2_scale = scale->r2_scale;
  const int c0 = blockIdx.y * COLS, cn = min(COLS, nc - c0);
  for (int i = tid; i < kFixTab; i += KFIX_THREADS) tab[i] = kFixExp2Tab[i];
  for (int i = tid; i < cn * (DP / 2); i += KFIX_THREADS)
    reinterpret_cast<int4 *>(su)[i] =
        reinterpret_cast<const int4 *>(ua + cols[c0 + i / (DP / 2)] * DP)[i % (DP / 2)];
  __syncthreads();
  const int64_t n = (int64_t)blockIdx.x * KFIX_THREADS + tid;
  if (n >= N) return;
  int2 u[DP];
  const int4 *src = reinterpret_cast<const int4 *>(ua + n * DP);
#pragma unroll
  for (int k = 0; k < DP; k += 2) {
    const int4 q = src[k / 2];
    u[k] = make_int2(q.x, q.y);
    u[k + 1] = make_int2(q.z, q.w);
  }
#pragma unroll 2
  for (int c = 0; c < cn; ++c)
    G[(int64_t)(c0 + c) * ldg + n] =
        fix_kappa<KERN, DP>(u, reinterpret_cast<const int4 *>(su[c]), fs, tab);
}

struct KmvFixArgs {
  const int2 *ur;
  int64_t Nr;
  const int2 *uc;
  const FixScale *scale;
  const double *V;
  int64_t ldv, N;
  int m;
  int64_t chunk;
  double *part;
};

template <int KERN, int DP>
cudaError_t launch_kmvfix_m(int M, dim3 grid, cudaStream_t s, const KmvFixArgs &a) {
  switch (M) {
#define KRR_CASE(MM)                                                                       \
  case MM:                                                                                 \
    kmvfix_kernel<KERN, DP, MM><<<grid, KFIX_THREADS, 0, s>>>(a.ur, a.Nr, a.uc, a.scale,    \
                                                             a.V, a.ldv, a.N, a.m, a.chunk, \
                                                             a.part);                      \
    break;
    KRR_CASE(1) KRR_CASE(2) KRR_CASE(4) KRR_CASE(8) KRR_CASE(16)
#undef KRR_CASE
    default:
      return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

#define KRR_FIX_DP_SWITCH(DP, FN, ...) \
  switch (DP) {                        \
    case 4: return FN<KERN, 4>(__VA_ARGS__);   \
    case 8: return FN<KERN, 8>(__VA_ARGS__);   \
    case 12: return FN<KERN, 12>(__VA_ARGS__); \
    case 16: return FN<KERN, 16>(__VA_ARGS__); \
    case 20: return FN<KERN, 20>(__VA_ARGS__); \
    case 24: return FN<KERN, 24>(__VA_ARGS__); \
    case 28: return FN<KERN, 28>(__VA_ARGS__); \
    case 32: return FN<KERN, 32>(__VA_ARGS__); \
    default: return cudaErrorInvalidValue;     \
  }

template <int KERN>
cudaError_t launch_kmvfix(int DP, int M, dim3 grid, cudaStream_t s, const KmvFixArgs &a) {
  KRR_FIX_DP_SWITCH(DP, launch_kmvfix_m, M, grid, s, a)
}

template <int KERN, int DP>
cudaError_t launch_kfix_columns_dp(const int2 *ua, int64_t N, const FixScale *scale,
                                   const int64_t *cols, int nc, double *G, int64_t ldg,
                                   cudaStream_t s) {
  kfix_columns_kernel<KERN, DP>
      <<<dim3((unsigned)ceil_div(N, KFIX_THREADS), (unsigned)ceil_div(nc, 32)), KFIX_THREADS, 0,
         s>>>(ua, N, scale, cols, nc, G, ldg);
  return cudaGetLastError();
}

template <int KERN>
cudaError_t launch_kfix_columns(int DP, const int2 *ua, int64_t N, const FixScale *scale,
                                const int64_t *cols, int nc, double *G, int64_t ldg,
                                cudaStream_t s) {
  KRR_FIX_DP_SWITCH(DP, launch_kfix_columns_dp, ua, N, scale, cols, nc, G, ldg, s)
}

}  // namespace krr
