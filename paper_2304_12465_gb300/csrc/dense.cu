// Dense building blocks of the k x k cores of Alg. 1 (lambda I + F^T F) and
// Alg. 2 (B^T B + H): Gram product, blocked float64 Cholesky and the inverse of
// its factor.
#include <algorithm>

#include "dense.cuh"

namespace krr {

// ------------------------------------------------------------ Gram (F^T F)
// Lower-triangular output tiles only; the terms go in chunks of GB_K through
// shared memory, the next chunk's on their way to registers meanwhile.
constexpr int GB_K = 16, G_THREADS = 256;
constexpr int GD_T = 64;               // float64: 64 x 64 tiles
constexpr int GF_M = 128, GF_N = 64;   // float32: 128 x 64 tiles,
constexpr int GF_K = 2 * GB_K;         // two chunks at a time

// Tile pair t of the lower triangle for tiles of M x N: row tile ti has the
// column tiles below (ti + 1) M.
template <int M, int N>
__device__ __forceinline__ void gram_tile(int t, int *ti, int *tj) {
  int i = 0;
  while (t >= (i + 1) * (M / N)) {
    t -= (i + 1) * (M / N);
    ++i;
  }
  *ti = i;
  *tj = t;
}

// Float64 throughout: a thread takes 4 x 4 entries.  Bound by the float64 pipe.
__global__ void __launch_bounds__(G_THREADS)
gram_lower_kernel(const double *__restrict__ F, int64_t N, int r, int kslice,
                  double *__restrict__ part) {
  __shared__ double As[GB_K][GD_T + 1];
  __shared__ double Bs[GB_K][GD_T + 1];
  int ti, tj;
  gram_tile<GD_T, GD_T>(blockIdx.x, &ti, &tj);
  const int tid = threadIdx.x, tx = tid % 16, ty = tid / 16;
  const int i0 = ti * GD_T, j0 = tj * GD_T;
  const int64_t kb = (int64_t)blockIdx.y * kslice;
  const int64_t ke = min(N, kb + kslice);
  double acc[4][4];
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int b = 0; b < 4; ++b) acc[a][b] = 0.0;
  for (int64_t k0 = kb; k0 < ke; k0 += GB_K) {
#pragma unroll
    for (int e = 0; e < (GD_T * GB_K) / G_THREADS; ++e) {
      const int idx = tid + e * G_THREADS;
      const int kk = idx % GB_K, ii = idx / GB_K;
      const int64_t gk = k0 + kk;
      As[kk][ii] = (i0 + ii < r && gk < ke) ? F[gk + (int64_t)(i0 + ii) * N] : 0.0;
      Bs[kk][ii] = (j0 + ii < r && gk < ke) ? F[gk + (int64_t)(j0 + ii) * N] : 0.0;
    }
    __syncthreads();
    double sum[4][4];
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
      for (int b = 0; b < 4; ++b) sum[a][b] = 0.0;
#pragma unroll
    for (int kk = 0; kk < GB_K; ++kk) {
      double av[4], bv[4];
#pragma unroll
      for (int a = 0; a < 4; ++a) av[a] = As[kk][ty + 16 * a];
#pragma unroll
      for (int b = 0; b < 4; ++b) bv[b] = Bs[kk][tx + 16 * b];
#pragma unroll
      for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) sum[a][b] = fma(av[a], bv[b], sum[a][b]);
    }
#pragma unroll
    for (int a = 0; a < 4; ++a)
#pragma unroll
      for (int b = 0; b < 4; ++b) acc[a][b] += sum[a][b];
    __syncthreads();
  }
  double *o = part + (int64_t)blockIdx.y * r * r;
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int b = 0; b < 4; ++b) {
      const int gi = i0 + ty + 16 * a, gj = j0 + tx + 16 * b;
      if (gi < r && gj <= gi) o[(int64_t)gi + (int64_t)gj * r] = acc[a][b];
    }
}

// float32 F: each chunk of GB_K products is summed in float32, then added to a
// float-float accumulator (Knuth's TwoSum, the rounding errors gathered in a
// float32 correction that is folded back every 8 chunks) -- float64 adds, at a
// small fraction of the float32 rate on this GPU, bounded the kernel.  A thread
// takes 8 x 4 entries as packed pairs of rows, so that three 16-byte loads
// serve 32 FMAs: with 4 x 4 entries and eight 4-byte loads the shared-memory
// wavefronts bound it (N = 1e5, r = 1000: 5.76 ms, now
// 4.23; 4.50 with one chunk at a time, 6.1 with two CTAs a SM and spills).
__global__ void __launch_bounds__(G_THREADS)
gram_lower_f32_kernel(const float *__restrict__ F, int64_t N, int r, int kslice,
                      double *__restrict__ part) {
  __shared__ __align__(16) float As[GF_K][GF_M + 4];
  __shared__ __align__(16) float Bs[GF_K][GF_N + 4];
  int ti, tj;
  gram_tile<GF_M, GF_N>(blockIdx.x, &ti, &tj);
  const int tid = threadIdx.x, tx = tid % 16, ty = tid / 16;
  const int i0 = ti * GF_M, j0 = tj * GF_N;
  const int64_t kb = (int64_t)blockIdx.y * kslice;
  const int64_t ke = min(N, kb + kslice);
  const float2 zero = make_float2(0.0f, 0.0f), minus = make_float2(-1.0f, -1.0f);
  float2 sh[4][4], sl[4][4];
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int b = 0; b < 4; ++b) sh[a][b] = sl[a][b] = zero;
  constexpr int NA = GF_M * GF_K / G_THREADS, NB = GF_N * GF_K / G_THREADS;
  constexpr int CS = G_THREADS / GF_K;
  float ra[NA], rb[NB];
  const int kk0 = tid % GF_K, ii0 = tid / GF_K;   // and every CS-th column from there
  auto load = [&](int64_t k0) {
    const int64_t gk = k0 + kk0;
#pragma unroll
    for (int e = 0; e < NA; ++e) {
      const int i = i0 + ii0 + CS * e;
      ra[e] = (i < r && gk < ke) ? F[gk + (int64_t)i * N] : 0.0f;
    }
#pragma unroll
    for (int e = 0; e < NB; ++e) {
      const int j = j0 + ii0 + CS * e;
      rb[e] = (j < r && gk < ke) ? F[gk + (int64_t)j * N] : 0.0f;
    }
  };
  // t = s + c with its rounding error (TwoSum); returns the error
  auto two_sum = [&](float2 &s, float2 c) {
    const float2 t = __fadd2_rn(s, c);
    const float2 z = __ffma2_rn(s, minus, t);
    const float2 u = __ffma2_rn(z, minus, t);
    const float2 err = __fadd2_rn(__ffma2_rn(u, minus, s), __ffma2_rn(z, minus, c));
    s = t;
    return err;
  };
  int chunk = 0;
  load(kb);
  for (int64_t k0 = kb; k0 < ke; k0 += GF_K) {
    __syncthreads();
#pragma unroll
    for (int e = 0; e < NA; ++e) As[kk0][ii0 + CS * e] = ra[e];
#pragma unroll
    for (int e = 0; e < NB; ++e) Bs[kk0][ii0 + CS * e] = rb[e];
    __syncthreads();
    if (k0 + GF_K < ke) load(k0 + GF_K);
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      float2 sum[4][4];
#pragma unroll
      for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) sum[a][b] = zero;
#pragma unroll
      for (int kk = 0; kk < GB_K; ++kk) {
        const float4 a0 = *reinterpret_cast<const float4 *>(&As[h * GB_K + kk][ty * 8]);
        const float4 a1 = *reinterpret_cast<const float4 *>(&As[h * GB_K + kk][ty * 8 + 4]);
        const float4 bq = *reinterpret_cast<const float4 *>(&Bs[h * GB_K + kk][tx * 4]);
        const float2 av[4] = {make_float2(a0.x, a0.y), make_float2(a0.z, a0.w),
                              make_float2(a1.x, a1.y), make_float2(a1.z, a1.w)};
        const float bv[4] = {bq.x, bq.y, bq.z, bq.w};
#pragma unroll
        for (int b = 0; b < 4; ++b)
#pragma unroll
          for (int a = 0; a < 4; ++a)
            sum[a][b] = __ffma2_rn(av[a], make_float2(bv[b], bv[b]), sum[a][b]);
      }
      ++chunk;
#pragma unroll
      for (int a = 0; a < 4; ++a)
#pragma unroll
        for (int b = 0; b < 4; ++b) {
          sl[a][b] = __fadd2_rn(sl[a][b], two_sum(sh[a][b], sum[a][b]));
          // fold the correction back, keeping it below an ulp of the sum
          if ((chunk & 7) == 0) sl[a][b] = two_sum(sh[a][b], sl[a][b]);
        }
    }
  }
  double *o = part + (int64_t)blockIdx.y * r * r;
#pragma unroll
  for (int a = 0; a < 4; ++a)
#pragma unroll
    for (int b = 0; b < 4; ++b) {
      const int gi = i0 + ty * 8 + 2 * a, gj = j0 + tx * 4 + b;
      if (gi < r && gj <= gi)
        o[(int64_t)gi + (int64_t)gj * r] = (double)sh[a][b].x + (double)sl[a][b].x;
      if (gi + 1 < r && gj <= gi + 1)
        o[(int64_t)gi + 1 + (int64_t)gj * r] = (double)sh[a][b].y + (double)sl[a][b].y;
    }
}

__global__ void gram_combine_kernel(const double *__restrict__ part, int slices, int r,
                                    double *__restrict__ C) {
  const int64_t total = (int64_t)r * r;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int i = (int)(e % r), j = (int)(e / r);
    if (j > i) continue;
    double acc = 0.0;
    for (int z = 0; z < slices; ++z) acc += part[(int64_t)z * total + e];
    C[e] = acc;
  }
}

template <typename T>
krr_status gram_lower(const T *F, int64_t N, int r, double *C, cudaStream_t s) {
  if (r <= 0) return KRR_OK;
  constexpr bool FLT = sizeof(T) == 4;
  constexpr int M = FLT ? GF_M : GD_T, RATIO = FLT ? GF_M / GF_N : 1;
  const int tiles = (r + M - 1) / M;
  const int ntri = tiles * (tiles + 1) / 2 * RATIO;   // a few beyond r or the diagonal
  // slices of the terms: float32 just under four waves of one CTA a SM, float64
  // two waves or more of two, down to 128 terms (r = 200, N = 4096: 40 CTAs
  // with slices of 1024 terms took 1127 us, 320 take 419)
  int64_t slices = ((int64_t)num_sms() * 4 + (FLT ? 0 : ntri - 1)) / ntri;
  slices = std::max<int64_t>(1, std::min<int64_t>(slices, FLT ? (N + 1023) / 1024 : (N + 127) / 128));
  int64_t kslice = (N + slices - 1) / slices;
  kslice = (kslice + GF_K - 1) / GF_K * GF_K;
  slices = (N + kslice - 1) / kslice;
  DevBuf<double> part;
  KRR_TRY(part.alloc((size_t)slices * r * r, s));
  const dim3 grid(ntri, (unsigned)slices);
  if constexpr (FLT)
    gram_lower_f32_kernel<<<grid, G_THREADS, 0, s>>>(F, N, r, (int)kslice, part.p);
  else
    gram_lower_kernel<<<grid, G_THREADS, 0, s>>>(F, N, r, (int)kslice, part.p);
  KRR_LAUNCH_CHECK();
  int blocks = ceil_div((int64_t)r * r, 256);
  if (blocks > num_sms() * 16) blocks = num_sms() * 16;
  gram_combine_kernel<<<blocks, 256, 0, s>>>(part.p, (int)slices, r, C);
  KRR_LAUNCH_CHECK();
  return KRR_OK;
}

template krr_status gram_lower<float>(const float *, int64_t, int, double *, cudaStream_t);
template krr_status gram_lower<double>(const double *, int64_t, int, double *, cudaStream_t);

// ------------------------------------------------------------ Cholesky
// Right-looking blocked Cholesky of the k x k cores.  The float64 pipe does
// 1.9 DFMA a clock on one SM, so what one block does alone is kept small: the
// diagonal block is 32 wide (11000 DFMA to factor and as many to invert it; a
// 64-wide one took 168 us), its inverse turns the panel's triangular solve
// into a product spread over the SMs by eight rows, and the trailing update
// touches the lower triangle only.
constexpr int CH_NB = 32;
constexpr int CH_PANEL_ROWS = 8;

// Factors the w x w diagonal block at A (lda) in place (lower; factor == 0:
// it already holds the factor) and writes the inverse of its factor to Dinv
// (CH_NB x CH_NB, column-major, zero padded).  blockIdx.x: block of a batch of
// diagonal blocks, CH_NB apart (n: size of the whole matrix).
__global__ void __launch_bounds__(128)
potrf_diag_kernel(double *__restrict__ A, int n, int64_t lda, double *__restrict__ Dinv,
                  int *__restrict__ status, int factor) {
  __shared__ double sA[CH_NB][CH_NB + 1], sW[CH_NB][CH_NB + 1], sR[CH_NB];
  __shared__ unsigned short order[CH_NB * (CH_NB + 1) / 2];
  const int o = blockIdx.x * CH_NB, w = min(CH_NB, n - o);
  A += o + (int64_t)o * lda;
  Dinv += (int64_t)blockIdx.x * CH_NB * CH_NB;
  const int tid = threadIdx.x, i = tid & 31, q = tid >> 5;
  for (int j = q; j < CH_NB; j += 4)
    sA[i][j] = (i < w && j < w && i >= j) ? A[i + (int64_t)j * lda] : (i == j ? 1.0 : 0.0);
  // the lower triangle's entries, last column first: those that the update of
  // column j touches are a prefix, which the threads share without idle lanes
  for (int j = q; j < CH_NB; j += 4) {
    const int m = CH_NB - 1 - j;   // entries of the columns after j
    if (i >= j) order[m * (m + 1) / 2 + (i - j)] = (unsigned short)(i << 8 | j);
  }
  __syncthreads();
  if (factor) {
    for (int j = 0; j < CH_NB; ++j) {
      if (q == 0) {
        const double p = sA[j][j];
        double d, r;
        sqrt_and_inverse(p, &d, &r);
        if (i == j) {
          if (!(p > 0.0)) atomicExch(status, 1);
          sA[j][j] = d;
          sR[j] = r;
        } else if (i > j) {
          const double x = sA[i][j], t = x * r;
          sA[i][j] = fma(fma(-t, d, x), r, t);
        }
      }
      __syncthreads();
      const int m = CH_NB - 1 - j, cnt = m * (m + 1) / 2;
      for (int e = tid; e < cnt; e += 128) {
        const int a = order[e] >> 8, c = order[e] & 255;
        sA[a][c] = fma(-sA[a][j], sA[c][j], sA[a][c]);
      }
      __syncthreads();
    }
    for (int j = q; j < w; j += 4)
      if (i >= j && i < w) A[i + (int64_t)j * lda] = sA[i][j];
  } else {
    if (tid < CH_NB) sR[tid] = 1.0 / sA[tid][tid];
    __syncthreads();
  }
  // inverse by forward substitution: four threads a column (partial sums of
  // every fourth term, added by shuffles)
  const int c = tid >> 2, t = tid & 3;
  for (int r = 0; r < CH_NB; ++r) {
    double v = 0.0;
    for (int l = c + t; l < r; l += 4) v = fma(-sA[r][l], sW[l][c], v);
    v += __shfl_xor_sync(0xffffffffu, v, 1);
    v += __shfl_xor_sync(0xffffffffu, v, 2);
    if (t == 0) sW[r][c] = r < c ? 0.0 : (r == c ? sR[r] : v * sR[r]);
    __syncwarp();
  }
  __syncthreads();
  for (int j = q; j < CH_NB; j += 4) Dinv[i + j * CH_NB] = (i < w && j < w) ? sW[i][j] : 0.0;
}

// A21 (r x w) <- A21 Dinv^T, eight rows a block.
__global__ void __launch_bounds__(256)
potrf_panel_kernel(double *__restrict__ A21, int r, int w, int64_t lda,
                   const double *__restrict__ Dinv) {
  __shared__ double sD[CH_NB][CH_NB + 1], sX[CH_PANEL_ROWS][CH_NB + 1];
  const int tid = threadIdx.x;
  for (int e = tid; e < CH_NB * CH_NB; e += 256) sD[e % CH_NB][e / CH_NB] = Dinv[e];
  const int row = tid & 7, j = tid >> 3;   // 8 rows x 32 columns
  const int i = blockIdx.x * CH_PANEL_ROWS + row;
  sX[row][j] = (i < r && j < w) ? A21[i + (int64_t)j * lda] : 0.0;
  __syncthreads();
  double v = 0.0;
#pragma unroll 8
  for (int l = 0; l < CH_NB; ++l) v = fma(sX[row][l], sD[j][l], v);   // Dinv is lower
  if (i < r && j < w) A21[i + (int64_t)j * lda] = v;
}

// A22 -= A21 A21^T on the lower triangle, 32 x 32 tiles (one a block).
__global__ void __launch_bounds__(256)
potrf_update_kernel(double *__restrict__ A21, int r, int w, int64_t lda) {
  __shared__ double sI[CH_NB][33], sJ[CH_NB][33];   // [column of A21][row]
  int t = blockIdx.x, ti = (int)((sqrtf(8.0f * t + 1.0f) - 1.0f) * 0.5f);
  while (ti * (ti + 1) / 2 > t) --ti;
  while ((ti + 1) * (ti + 2) / 2 <= t) ++ti;
  const int tj = t - ti * (ti + 1) / 2;
  const int tid = threadIdx.x;
  for (int e = tid; e < CH_NB * 32; e += 256) {
    const int l = e >> 5, x = e & 31;
    const int i = ti * 32 + x, j = tj * 32 + x;
    sI[l][x] = (i < r && l < w) ? A21[i + (int64_t)l * lda] : 0.0;
    sJ[l][x] = (j < r && l < w) ? A21[j + (int64_t)l * lda] : 0.0;
  }
  __syncthreads();
  double *A22 = A21 + (int64_t)w * lda;
  const int x = tid & 31, y = tid >> 5;   // row x, columns y + 8 u
  double acc[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll 8
  for (int l = 0; l < CH_NB; ++l) {
    const double a = sI[l][x];
#pragma unroll
    for (int u = 0; u < 4; ++u) acc[u] = fma(a, sJ[l][y + 8 * u], acc[u]);
  }
  const int i = ti * 32 + x;
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const int j = tj * 32 + y + 8 * u;
    if (i < r && j <= i) A22[i + (int64_t)j * lda] -= acc[u];
  }
}

krr_status potrf_lower(double *A, int n, int64_t lda, cudaStream_t s) {
  if (n <= 0) return KRR_OK;
  DevBuf<int> status;
  KRR_TRY(status.alloc(1, s));
  KRR_CUDA_TRY(cudaMemsetAsync(status.p, 0, sizeof(int), s));
  DevBuf<double> dinv;
  KRR_TRY(dinv.alloc(CH_NB * CH_NB, s));
  for (int o = 0; o < n; o += CH_NB) {
    const int w = std::min(CH_NB, n - o);
    double *Abb = A + o + (int64_t)o * lda;
    potrf_diag_kernel<<<1, 128, 0, s>>>(Abb, w, lda, dinv.p, status.p, 1);
    KRR_LAUNCH_CHECK();
    const int r = n - o - w;
    if (r <= 0) break;
    potrf_panel_kernel<<<ceil_div(r, CH_PANEL_ROWS), 256, 0, s>>>(Abb + w, r, w, lda, dinv.p);
    KRR_LAUNCH_CHECK();
    const int tiles = (r + 31) / 32;
    potrf_update_kernel<<<tiles * (tiles + 1) / 2, 256, 0, s>>>(Abb + w, r, w, lda);
    KRR_LAUNCH_CHECK();
  }
  int h = 0;
  KRR_CUDA_TRY(cudaMemcpyAsync(&h, status.p, sizeof(int), cudaMemcpyDeviceToHost, s));
  KRR_CUDA_TRY(cudaStreamSynchronize(s));
  if (h) {
    set_error("Cholesky factorisation met a non-positive pivot (matrix not numerically "
              "positive definite)");
    return KRR_ECHOL;
  }
  return KRR_OK;
}

// W <- the inverses of the diagonal blocks, zero elsewhere.
__global__ void trinv_init_kernel(const double *__restrict__ Dinv, int n, double *__restrict__ W) {
  const int64_t total = (int64_t)n * n;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int j = (int)(e / n), i = (int)(e - (int64_t)j * n);
    const int b = i / CH_NB;
    W[e] = (b == j / CH_NB)
               ? Dinv[(int64_t)b * CH_NB * CH_NB + (i - b * CH_NB) + (j - b * CH_NB) * CH_NB]
               : 0.0;
  }
}

// One half of a doubling step of the inverse: the pairs of size-h diagonal
// blocks (rows p 2h .. of the first, + h of the second) whose inverses W holds.
//   first  half: T21 = L21 W11          (columns of W11 are lower: k >= column)
//   second half: W21 = -W22 T21         (rows of W22 are lower: k <= row)
// T (n x n, only the blocks below the pairs' diagonals) is scratch.  A block
// does a 32 x 32 tile over the k that are not zero.
template <bool FIRST>
__global__ void __launch_bounds__(256)
trinv_level_kernel(const double *__restrict__ L, int64_t lda, int n, int h, double *__restrict__ W,
                   double *__restrict__ T) {
  __shared__ double sX[32][33], sY[32][33];   // [k][row], [k][column]
  const int o = blockIdx.z * 2 * h;            // first row of the pair
  const int r0 = o + h + blockIdx.x * 32, c0 = o + blockIdx.y * 32;
  if (r0 >= n) return;
  const int rows = min(o + 2 * h, n);
  const int tid = threadIdx.x, x = tid & 31, y = tid >> 5;
  double acc[4] = {0.0, 0.0, 0.0, 0.0};
  const int kb = FIRST ? c0 : o + h, ke = FIRST ? o + h : min(r0 + 32, rows);
  for (int k0 = kb; k0 < ke; k0 += 32) {
    __syncthreads();
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int kk = y + 8 * u, k = k0 + kk;
      // X(row, k): contiguous in rows; Y(k, column): contiguous in k
      double a = 0.0, b = 0.0;
      if (r0 + x < rows && k < ke)
        a = FIRST ? L[r0 + x + (int64_t)k * lda] : W[r0 + x + (int64_t)k * n];
      const int kx = k0 + x;
      if (kx < ke) b = FIRST ? W[kx + (int64_t)(c0 + kk) * n] : T[kx + (int64_t)(c0 + kk) * n];
      sX[kk][x] = a;
      sY[x][kk] = b;
    }
    __syncthreads();
#pragma unroll 8
    for (int l = 0; l < 32; ++l) {
      const double a = sX[l][x];
#pragma unroll
      for (int u = 0; u < 4; ++u) acc[u] = fma(a, sY[l][y + 8 * u], acc[u]);
    }
  }
  if (r0 + x < rows)
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int64_t e = r0 + x + (int64_t)(c0 + y + 8 * u) * n;
      if (FIRST) T[e] = acc[u];
      else W[e] = -acc[u];
    }
}

// Inverse by doubling: the diagonal blocks' inverses (one launch), then pairs
// of inverted blocks of 32, 64, ... joined by two products a level, all pairs
// of a level in one launch.  Row by row of blocks (each row a product with
// everything before it) it was a chain of small grids: 30 launches and 9 ms at
// n = 1000.
krr_status trinv_lower(const double *L, int n, int64_t lda, double *W, cudaStream_t s) {
  if (n <= 0) return KRR_OK;
  const int nb = (n + CH_NB - 1) / CH_NB;
  DevBuf<double> dinv, T;
  KRR_TRY(dinv.alloc((size_t)nb * CH_NB * CH_NB, s));
  KRR_TRY(T.alloc((size_t)n * n, s));
  potrf_diag_kernel<<<nb, 128, 0, s>>>(const_cast<double *>(L), n, lda, dinv.p, nullptr, 0);
  KRR_LAUNCH_CHECK();
  const int64_t g = std::min<int64_t>(((int64_t)n * n + 255) / 256, (int64_t)num_sms() * 16);
  trinv_init_kernel<<<(unsigned)g, 256, 0, s>>>(dinv.p, n, W);
  KRR_LAUNCH_CHECK();
  for (int h = CH_NB; h < n; h *= 2) {
    const int pairs = (n - h + 2 * h - 1) / (2 * h);   // pairs with a second block
    const dim3 grid(h / 32, h / 32, pairs);
    trinv_level_kernel<true><<<grid, 256, 0, s>>>(L, lda, n, h, W, T.p);
    KRR_LAUNCH_CHECK();
    trinv_level_kernel<false><<<grid, 256, 0, s>>>(L, lda, n, h, W, T.p);
    KRR_LAUNCH_CHECK();
  }
  return KRR_OK;
}

__global__ void add_diag_kernel(double *A, int n, int64_t lda, double v) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) A[i + (int64_t)i * lda] += v;
}

krr_status add_diagonal(double *A, int n, int64_t lda, double v, cudaStream_t s) {
  if (n <= 0) return KRR_OK;
  add_diag_kernel<<<ceil_div(n, 256), 256, 0, s>>>(A, n, lda, v);
  KRR_LAUNCH_CHECK();
  return KRR_OK;
}

__global__ void transpose_kernel(const double *__restrict__ A, int n, double *__restrict__ B) {
  __shared__ double tile[32][33];
  const int bx = blockIdx.x * 32, by = blockIdx.y * 32;
  for (int j = threadIdx.y; j < 32; j += blockDim.y) {
    const int r = bx + threadIdx.x, c = by + j;
    if (r < n && c < n) tile[j][threadIdx.x] = A[r + (int64_t)c * n];
  }
  __syncthreads();
  for (int j = threadIdx.y; j < 32; j += blockDim.y) {
    const int r = by + threadIdx.x, c = bx + j;
    if (r < n && c < n) B[r + (int64_t)c * n] = tile[threadIdx.x][j];
  }
}

krr_status transpose_square(const double *A, int n, double *B, cudaStream_t s) {
  if (n <= 0) return KRR_OK;
  dim3 grid((n + 31) / 32, (n + 31) / 32), block(32, 8);
  transpose_kernel<<<grid, block, 0, s>>>(A, n, B);
  KRR_LAUNCH_CHECK();
  return KRR_OK;
}

}  // namespace krr
