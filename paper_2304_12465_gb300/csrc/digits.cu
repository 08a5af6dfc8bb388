// C -= A B^T by digits on the fp16 tensor cores (digits.cuh): the Schur update
// of Alg. 3 and the off-diagonal part of its triangular solve.
#include <algorithm>

#include "dense.cuh"
#include "digits.cuh"

namespace krr {

constexpr int DG_THREADS = 256;
constexpr int DG_ROWS = 64;        // rows of C per CTA: four 16-row tiles
constexpr int DG_STAGES = 4;       // ring of B digits: two pairs of steps
constexpr int DG_KSTEPS = DIG_CHUNK / 16;

__device__ __forceinline__ void dg_mma(float (&c)[4], const uint4 &a, const uint2 &b) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, "
      "{%8,%9}, {%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a.x), "r"(a.y), "r"(a.z), "r"(a.w), "r"(b.x), "r"(b.y));
}

// Digits of B (nc rows of K entries: row c at B + rows[c] (rows NULL: c), step
// ldb between entries) as MMA B fragments, zero padded to K16 steps of 16 and
// NT tiles of 8 rows: frag[((step NT + tile) 7 + digit) 32 + lane].
__global__ void dig_rows_kernel(const double *__restrict__ B, int64_t ldb,
                                const int64_t *__restrict__ rows, int nc, int K, int K16, int NT, uint2 *__restrict__ frag) {
  const int64_t total = (int64_t)K16 * NT * 32;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int lane = (int)(e & 31), tile = (int)((e >> 5) % NT);
    const int step = (int)((e >> 5) / NT);
    const int c = tile * 8 + (lane >> 2), k = step * 16 + 2 * (lane & 3);
    double x[4] = {0.0, 0.0, 0.0, 0.0};
    if (c < nc) {
      const int64_t r = rows ? rows[c] : c;
#pragma unroll
      for (int t = 0; t < 4; ++t) {
        const int kk = k + (t & 1) + 8 * (t >> 1);
        if (kk < K) x[t] = B[r + (int64_t)kk * ldb];
      }
    }
    uint32_t d0[DIG_N], d1[DIG_N];
    dig_pair(x[0], x[1], d0);
    dig_pair(x[2], x[3], d1);
    uint2 *dst = frag + ((int64_t)(step * NT + tile) * DIG_N) * 32 + lane;
#pragma unroll
    for (int s = 0; s < DIG_N; ++s) dst[s * 32] = make_uint2(d0[s], d1[s]);
  }
}

// C (N x nc, ldc) -= A (N x K, lda) B^T, B as fragments; cmap (optional) gives
// the column of C for each row of B.  A CTA takes 64 rows
// and all columns; warp (r, h) the 16 rows of tile r and NTW column tiles of
// half h.  Per step of 16 terms each warp converts its half of its row tile's
// entries (read column by column, 64-byte segments), the two halves meet in
// shared memory as MMA A fragments, and B fragments arrive through a ring of
// asynchronous copies.  Tensor bound: 28 MMAs a tile and step against about
// 30 other instructions.  The accumulators (28 floats a tile) set NTW <= 7
// and one CTA a SM.  Measured at N = 1e5, 100 columns: 1.04 ms for K = 500 and
// 1.75 ms for K = 900, against 3.35 and 5.87 ms for a float-float product on
// the float32 pipe (3.3 clocks an MMA where the pipe's best is 2.1: eight
// warps a SM do not fill it, and converting inside the MMA sequence spilled
// and took 2.48 ms).
template <int NTW>
__global__ void __launch_bounds__(DG_THREADS, 1)
dig_gemm_kernel(const double *__restrict__ A, int64_t lda, int64_t N, int K,
                const uint2 *__restrict__ frag, int nc, double *__restrict__ C, int64_t ldc,
                const int *__restrict__ cmap) {
  constexpr int NT = 2 * NTW;
  constexpr int BSTEP = NT * DIG_N * 32;                 // uint2 of one step
  extern __shared__ __align__(16) unsigned char dg_smem[];
  uint2 *sB = reinterpret_cast<uint2 *>(dg_smem);        // [DG_STAGES][BSTEP]
  uint4 *sA = reinterpret_cast<uint4 *>(sB + DG_STAGES * BSTEP);   // [2][4][DIG_N][32]
  int64_t *tot = reinterpret_cast<int64_t *>(sA + 2 * 4 * DIG_N * 32);   // [NTW 4][256]
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int rt = warp >> 1, half = warp & 1;
  const int g = lane >> 2, q = lane & 3;
  const int64_t r0 = (int64_t)blockIdx.x * DG_ROWS + rt * 16 + g;
  const bool ok0 = r0 < N, ok1 = r0 + 8 < N;
  const int steps = (K + 15) / 16;

  auto load_a = [&](int step, double (&x)[4]) {
    const int k = step * 16 + half * 8 + 2 * q;
    const double *p = A + r0 + (int64_t)k * lda;
    x[0] = (ok0 && k < K) ? p[0] : 0.0;
    x[1] = (ok0 && k + 1 < K) ? p[lda] : 0.0;
    x[2] = (ok1 && k < K) ? p[8] : 0.0;
    x[3] = (ok1 && k + 1 < K) ? p[lda + 8] : 0.0;
  };
  auto copy_b = [&](int step) {
    if (step < steps) {
      const char *src = reinterpret_cast<const char *>(frag + (int64_t)step * BSTEP);
      const uint32_t dst =
          (uint32_t)__cvta_generic_to_shared(sB + (step % DG_STAGES) * BSTEP);
      for (int i = tid; i < BSTEP / 2; i += DG_THREADS)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + i * 16),
                     "l"(src + i * 16));
    }
  };

  float acc[NTW][DIG_N][4];
#pragma unroll
  for (int j = 0; j < NTW; ++j)
#pragma unroll
    for (int s = 0; s < DIG_N; ++s)
#pragma unroll
      for (int e = 0; e < 4; ++e) acc[j][s][e] = 0.0f;
#pragma unroll
  for (int j = 0; j < NTW * 4; ++j) tot[j * DG_THREADS + tid] = 0;

  double x[4];
  auto store_a = [&](int step) {
    uint2 *dst = reinterpret_cast<uint2 *>(sA + ((step & 1) * 4 + rt) * DIG_N * 32 + lane) + half;
    uint32_t d0[DIG_N], d1[DIG_N];
    dig_pair(x[0], x[1], d0);
    dig_pair(x[2], x[3], d1);
#pragma unroll
    for (int s = 0; s < DIG_N; ++s) dst[s * 64] = make_uint2(d0[s], d1[s]);
  };
  load_a(0, x);
  copy_b(0);
  copy_b(1);
  for (int step = 0; step < steps; ++step) {
    store_a(step);
    if ((step & 1) == 0) {
      // a pair of steps of B has arrived, and every warp is done with the
      // pair before it, whose place the next pair takes
      asm volatile("cp.async.wait_all;" ::: "memory");
      __syncthreads();
      copy_b(step + 2);
      copy_b(step + 3);
    } else {
      // only the two warps of a row tile share its digits, so that the row
      // tiles' conversions and MMAs drift apart and overlap
      asm volatile("bar.sync %0, 64;" ::"r"(rt + 1) : "memory");
    }
    if (step + 1 < steps) load_a(step + 1, x);
    const uint4 *bufA = sA + ((step & 1) * 4 + rt) * DIG_N * 32;
    uint4 a[DIG_N];
#pragma unroll
    for (int s = 0; s < DIG_N; ++s) a[s] = bufA[s * 32 + lane];
    const uint2 *bufB = sB + (step % DG_STAGES) * BSTEP + half * NTW * DIG_N * 32 + lane;
#pragma unroll
    for (int j = 0; j < NTW; ++j)
#pragma unroll
      for (int t = 0; t < DIG_N; ++t) {
        const uint2 b = bufB[(j * DIG_N + t) * 32];
#pragma unroll
        for (int s = 0; s + t < DIG_N; ++s) dg_mma(acc[j][s + t], a[s], b);
      }
    if ((step + 1) % DG_KSTEPS == 0 || step + 1 == steps) {
#pragma unroll
      for (int j = 0; j < NTW; ++j)
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          // units 2^-32 and 2^-64, both exact
          const int64_t hi = ((int64_t)__float2int_rn(acc[j][0][e]) << 16) +
                             ((int64_t)__float2int_rn(acc[j][1][e]) << 8) +
                             (int64_t)__float2int_rn(acc[j][2][e]);
          const int64_t lo = ((int64_t)__float2int_rn(acc[j][3][e]) << 24) +
                             ((int64_t)__float2int_rn(acc[j][4][e]) << 16) +
                             ((int64_t)__float2int_rn(acc[j][5][e]) << 8) +
                             (int64_t)__float2int_rn(acc[j][6][e]);
          tot[(j * 4 + e) * DG_THREADS + tid] += hi * (1ll << 28) + ((lo + 8) >> 4);
#pragma unroll
          for (int s = 0; s < DIG_N; ++s) acc[j][s][e] = 0.0f;
        }
    }
  }
#pragma unroll
  for (int j = 0; j < NTW; ++j)
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int c = (half * NTW + j) * 8 + 2 * q + (e & 1);
      const bool ok = (e >> 1) ? ok1 : ok0;
      if (ok && c < nc) {
        double *dst = C + r0 + (e >> 1) * 8 + (int64_t)(cmap ? cmap[c] : c) * ldc;
        *dst -= (double)tot[(j * 4 + e) * DG_THREADS + tid] * 0x1p-60;
      }
    }
}

static size_t dig_smem(int NTW) {
  return (size_t)DG_STAGES * 2 * NTW * DIG_N * 32 * sizeof(uint2) +
         (size_t)2 * 4 * DIG_N * 32 * sizeof(uint4) +
         (size_t)NTW * 4 * DG_THREADS * sizeof(int64_t);
}

template <int NTW>
static krr_status launch_dig(const double *A, int64_t lda, int64_t N, int K, const uint2 *frag,
                             int nc, double *C, int64_t ldc, const int *cmap, cudaStream_t s) {
  const size_t smem = dig_smem(NTW);
  KRR_TRY(raise_smem_limit(dig_gemm_kernel<NTW>, smem));
  dig_gemm_kernel<NTW><<<ceil_div(N, DG_ROWS), DG_THREADS, smem, s>>>(A, lda, N, K, frag, nc, C,
                                                                     ldc, cmap);
  KRR_LAUNCH_CHECK();
  return KRR_OK;
}

// Column tiles of a warp: half of the columns, rounded up to an instance.
static int dig_ntw(int nc) {
  const int tiles = (nc + 7) / 8;
  return tiles <= 2 ? 1 : tiles <= 4 ? 2 : tiles <= 8 ? 4 : 7;
}

size_t dig_frag_elems(int nc, int K) {
  return (size_t)((K + 15) / 16) * 2 * dig_ntw(std::min(nc, DIG_MAX_COLS)) * DIG_N * 32;
}

krr_status dig_gemm_sub(const double *A, int64_t lda, int64_t N, int K, const double *B,
                        int64_t ldb, const int64_t *rows, int nc, double *C, int64_t ldc,
                        const int *cmap, uint2 *frag, cudaStream_t s) {
  if (N <= 0 || K <= 0 || nc <= 0) return KRR_OK;
  for (int c0 = 0; c0 < nc; c0 += DIG_MAX_COLS) {
    const int n = std::min(DIG_MAX_COLS, nc - c0);
    const int NTW = dig_ntw(n);
    const int K16 = (K + 15) / 16;
    const int64_t total = (int64_t)K16 * 2 * NTW * 32;
    dig_rows_kernel<<<(unsigned)std::min<int64_t>((total + 127) / 128, 4 * num_sms()), 128, 0,
                      s>>>(rows ? B : B + c0, ldb, rows ? rows + c0 : nullptr, n, K, K16, 2 * NTW, frag);
    KRR_LAUNCH_CHECK();
    double *Cc = cmap ? C : C + (int64_t)c0 * ldc;
    const int *cm = cmap ? cmap + c0 : nullptr;
    switch (NTW) {
      case 1: KRR_TRY(launch_dig<1>(A, lda, N, K, frag, n, Cc, ldc, cm, s)); break;
      case 2: KRR_TRY(launch_dig<2>(A, lda, N, K, frag, n, Cc, ldc, cm, s)); break;
      case 4: KRR_TRY(launch_dig<4>(A, lda, N, K, frag, n, Cc, ldc, cm, s)); break;
      default: KRR_TRY(launch_dig<7>(A, lda, N, K, frag, n, Cc, ldc, cm, s)); break;
    }
  }
  return KRR_OK;
}

}  // namespace krr
