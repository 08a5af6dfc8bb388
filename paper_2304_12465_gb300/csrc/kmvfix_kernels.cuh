// Float64 and float-float products and float64 kernel columns on fixed-point
// kernel values (kfix.cuh).
//
// The integer multiplies bound them (the FMA pipe's heavy half, which they
// share, is 80% busy at d = 8): per entry 3d multiply-adds for the sums of
// squares (2d float-float) plus about 15 for 2^-E, then one DFMA per
// right-hand side (1.9 a clock and SM) or 12 float32 operations.  A thread
// keeps two rows' limbs in registers (one for d > 16, where two would spill)
// and walks a shared tile of columns, which every lane reads at the same
// address.  Square products of few right-hand sides evaluate each pair of
// points once (kmvfixsym_kernel).  Measured, Gaussian, one right-hand side:
// N = 4096, d = 8 float64 123 us, symmetric 88 us (1055 us for kmv64_kernel);
// four right-hand sides: N = 40000, d = 16 float-float 16.0 ms, symmetric 10.15
// ms (14.1 ms for kmvffsym_kernel).  20 kernel columns at N = 4096: 7.3 us
// against 34.7 in float64 arithmetic.
#pragma once

#include "kfix.cuh"
#include "kmv.cuh"
#include "kmvff_kernels.cuh"

namespace krr {

constexpr int KFIX_THREADS = 128;
constexpr int KFIX_TJ = 32;

__host__ __device__ constexpr int kmvfix_rows_per_thread(int DP) { return DP <= 16 ? 2 : 1; }

// ------------------------------------------------ the two accumulations
// Float64 values and sums (one DFMA a right-hand side), or float-float ones
// (12 float32 operations; 128 a clock and SM against 1.9).
struct FixAccD {
  using T = double;
  static constexpr bool kFF = false;
  static __device__ __forceinline__ T zero() { return 0.0; }
  static __device__ __forceinline__ T load(double v) { return v; }
  static __device__ __forceinline__ void fma_(T &acc, T k, T v) { acc = fma(k, v, acc); }
  static __device__ __forceinline__ T add(T a, T b) { return a + b; }
  static __device__ __forceinline__ double value(T a) { return a; }
};
struct FixAccFF {
  using T = FF;
  static constexpr bool kFF = true;
  static __device__ __forceinline__ T zero() { return {0.0f, 0.0f}; }
  static __device__ __forceinline__ T load(double v) {
    const float h = (float)v;
    return {h, (float)(v - (double)h)};
  }
  static __device__ __forceinline__ void fma_(T &acc, T k, T v) { ff_fma_acc(acc, k, v.h, v.l); }
  static __device__ __forceinline__ T add(T a, T b) { return ff_add(a, b); }
  static __device__ __forceinline__ double value(T a) { return (double)a.h + (double)a.l; }
};

// 2^-E as hi + lo floats: 24 bits rounded to nearest and the signed rest (32
// bits, rounded to 24 by the conversion), 49 bits of the mantissa or more.
__device__ __forceinline__ FF fix_exp2_ff(uint64_t E, const uint64_t *__restrict__ tab) {
  const int n = (int)(E >> 54);
  // m in [2^62, 2^63]: hi from bit 39 up, rounded by half its unit, 2^38 (bit 63
  // carries into the exponent field); lo the 32 bits below in units of 2^-56, whose
  // top bit, set where hi was rounded up, makes them negative
  const uint64_t m = fix_exp2_mantissa(E, tab);
  const float h =
      __uint_as_float(0x4B000000u + ((((uint32_t)(m >> 32) + 64u) >> 7) - 0x800000u));
  const float l = (float)(int32_t)(uint32_t)(m >> 7);
  if (n < 64) {
    const float s = __uint_as_float((uint32_t)(127 - 24 - n) << 23);   // 2^(-24 - n)
    return {h * s, l * (s * 0x1p-32f)};
  }
  // down to the smallest float, both parts (subnormal ones rounded once)
  if (n > 150) return {0.0f, 0.0f};
  const float s = __uint_as_float((uint32_t)(127 + 40 - n) << 23);     // 2^(40 - n)
  return {(h * 0x1p-64f) * s, (l * 0x1p-96f) * s};
}

// The squared distance 2^(26 - 2 q) (2^24 S1 + A) as a float-float value (its
// leading 48 bits or more).
__device__ __forceinline__ FF fix_r2_ff(int64_t S1, int64_t A, int q) {
  uint64_t lo = (uint64_t)S1 << 24;
  int64_t hi = S1 >> 40;
  const uint64_t t = lo + (uint64_t)A;
  hi += (A >> 63) + (t < lo ? 1 : 0);
  lo = t;
  if (hi < 0 || (hi == 0 && lo == 0)) return {0.0f, 0.0f};   // see fix_exponent_ff
  int ex;
  uint64_t top;
  if (hi) {
    const int lz = __clzll(hi);
    top = lz ? ((uint64_t)hi << lz) | (lo >> (64 - lz)) : (uint64_t)hi;
    ex = 128 - lz;
  } else {
    const int lz = __clzll((long long)lo);
    top = lo << lz;
    ex = 64 - lz;
  }
  // value = top 2^(ex - 64) 2^(26 - 2 q), top in [2^63, 2^64)
  const float h = __uint_as_float(0x4B000000u + ((uint32_t)(top >> 40) - 0x800000u));
  const float l = (float)(uint32_t)(top >> 8);
  const int e2 = ex - 24 + 26 - 2 * q;                                  // exponent of h's unit
  const float s = __uint_as_float((uint32_t)max(127 + e2, 1) << 23);
  return {h * s, (l * s) * 0x1p-32f};
}

// kappa of one pair from the row's coordinates (registers) and the column's
// (shared, 16-byte aligned); cst: the constants of exp_ff (Matern, float-float).
template <typename A, int KERN, int DP>
__device__ __forceinline__ typename A::T fix_kappa(const int2 (&u)[DP],
                                                   const int4 *__restrict__ v,
                                                   const FixScale &fs,
                                                   const uint64_t *__restrict__ tab,
                                                   const float *__restrict__ cst) {
  if constexpr (KERN == KLAPLACE) {
    // the float64 sums of more than one group of coordinates keep their lowest bits
    constexpr bool GROUPS = DP > kFixL1Group && !A::kFF;
    uint64_t S = 0, G = 0;   // sums of the groups before without their low bits
    uint32_t L = 0;          // (those apart), and of the present one
#pragma unroll
    for (int k = 0; k < DP; k += 2) {
      const int4 b = v[k / 2];
      const int64_t d0 = (int64_t)(((uint64_t)(uint32_t)u[k].y << 32) | (uint32_t)u[k].x) -
                         (int64_t)(((uint64_t)(uint32_t)b.y << 32) | (uint32_t)b.x);
      const int64_t d1 = (int64_t)(((uint64_t)(uint32_t)u[k + 1].y << 32) | (uint32_t)u[k + 1].x) -
                         (int64_t)(((uint64_t)(uint32_t)b.w << 32) | (uint32_t)b.z);
      G += (uint64_t)llabs(d0) + (uint64_t)llabs(d1);
      if constexpr (GROUPS)
        if ((k + 2) % kFixL1Group == 0 || k + 2 == DP) {
          S += G >> kFixL1Low;
          L += (uint32_t)G & ((1u << kFixL1Low) - 1);
          G = 0;
        }
    }
    const uint64_t E = GROUPS ? fix_exponent_l1_groups(S, L, fs.r - kFixL1Low)
                              : fix_exponent_l1(G, fs.r);
    if constexpr (A::kFF) return fix_exp2_ff(E, tab);
    else return fix_exp2(E, tab);
  } else {
    int64_t S1 = 0, S2 = A::kFF ? fs.bias : 0;
    uint64_t S3 = 0;
#pragma unroll
    for (int k = 0; k < DP; k += 2) {
      const int4 b = v[k / 2];
      const int h0 = u[k].x - b.x, l0 = u[k].y - b.y;
      const int h1 = u[k + 1].x - b.z, l1 = u[k + 1].y - b.w;
      S1 += (int64_t)h0 * h0;
      S2 += (int64_t)h0 * l0;
      S1 += (int64_t)h1 * h1;
      S2 += (int64_t)h1 * l1;
      if constexpr (!A::kFF) {
        S3 += (uint64_t)((int64_t)l0 * l0);
        S3 += (uint64_t)((int64_t)l1 * l1);
      }
    }
    if constexpr (A::kFF) {
      // near points (few in most sets) take the squares of their low limbs in place
      // of the mean; S1 is not negative.  Measured against no near points, N =
      // 40000, d = 16, m = 4: 9.8 -> 10.2 ms; with the mean added here and a 64-bit
      // comparison 10.4; with the branch after two pairs, or a tile repeated when it
      // holds a near pair, 10.1 to 10.8 and up to 1.4 times as much in dense sets
      if ((uint32_t)(S1 >> 32) < fs.s1_near) {
#pragma unroll
        for (int k = 0; k < DP; k += 2) {
          const int4 b = v[k / 2];
          const int l0 = u[k].y - b.y, l1 = u[k + 1].y - b.w;
          S3 += (uint64_t)((int64_t)l0 * l0);
          S3 += (uint64_t)((int64_t)l1 * l1);
        }
        S2 += (int64_t)(S3 >> 26) - fs.bias;
      }
      if constexpr (KERN == KMATERN) {
        const FF q = sqrt_ff(fix_r2_ff(S1, S2, fs.q));
        const FF e = exp_ff({-q.h, -q.l}, cst, cst + 4);
        const FF third = {0.3333333433f, -9.9341077e-09f};
        return ff_mul(ff_add({1.0f, 0.0f}, ff_add(q, ff_mul(ff_mul(q, q), third))), e);
      } else {
        return fix_exp2_ff(fix_exponent_ff(S1, S2, fs.r, fs.s1_max), tab);
      }
    } else if constexpr (KERN == KMATERN) {
      return fix_matern(S1, S2, S3, fs.r2_scale, tab);
    } else {
      return fix_exp2(fix_exponent(S1, S2, S3, fs.r, fs.s1_max), tab);
    }
  }
}

// The scale and the tables of a CTA: exp2 table and, for the Matern float-float
// values, exp_ff's constants.
__device__ __forceinline__ FixScale fix_load_scale(const FixScale *__restrict__ scale) {
  FixScale fs;
  fs.r = scale->r;
  fs.q = scale->q;
  fs.s1_max = scale->s1_max;
  fs.r2_scale = scale->r2_scale;
  fs.bias = scale->bias;
  fs.s1_near = scale->s1_near;
  return fs;
}
template <typename A, int KERN>
__device__ __forceinline__ void fix_load_tables(const ExpFFConsts &ec, uint64_t *tab, float *cst) {
  for (int i = threadIdx.x; i < kFixTab; i += KFIX_THREADS) tab[i] = kFixExp2Tab[i];
  if constexpr (KERN == KMATERN && A::kFF) {
    if (threadIdx.x < 4) cst[threadIdx.x] = ec.c[threadIdx.x];
    if (threadIdx.x < 64) cst[4 + threadIdx.x] = ec.tab[threadIdx.x];
  }
}

// CTAs a SM that a rectangular product of one or two right-hand sides keeps room
// for (1: the compiler's choice).  The branch of the float-float near pairs takes 8
// to 36 registers more than the rest and would cost one or two of them: 4e5 points,
// one right-hand side, 2000 columns, d = 20: 8.30 ms, 7.96 with the limit (7.75
// without near pairs); 1000 columns, d = 16: 3.73 and 3.47.
__host__ __device__ constexpr int kmvfix_min_ctas(bool ff, int DP, int M) {
  if (!ff || M > 2 || DP <= 4) return 1;
  return DP <= 8 ? 7 : DP <= 16 ? 4 : DP <= 20 ? 7 : DP <= 24 ? 6 : 5;
}

// part[split][c][row] = sum over the split's columns of kappa v; ur (Nr x DP),
// uc (N x DP): coordinates of rows and columns.
template <typename A, int KERN, int DP, int M>
__global__ void __launch_bounds__(KFIX_THREADS, kmvfix_min_ctas(A::kFF, DP, M))
kmvfix_kernel(const int2 *__restrict__ ur, int64_t Nr, const int2 *__restrict__ uc,
              const FixScale *__restrict__ scale, const double *__restrict__ V, int64_t ldv,
              int64_t N, int m, int64_t chunk, const ExpFFConsts ec, double *__restrict__ part) {
  using T = typename A::T;
  constexpr int RI = kmvfix_rows_per_thread(DP);
  __shared__ __align__(16) int2 su[KFIX_TJ][DP];
  __shared__ __align__(16) T sv[KFIX_TJ][M];
  __shared__ uint64_t tab[kFixTab];
  __shared__ float cst[KERN == KMATERN && A::kFF ? 68 : 1];
  if (!scale->ok) return;
  const int tid = threadIdx.x;
  const FixScale fs = fix_load_scale(scale);
  fix_load_tables<A, KERN>(ec, tab, cst);
  const int64_t row0 = (int64_t)blockIdx.x * (KFIX_THREADS * RI) + tid;
  const int64_t j_begin = (int64_t)blockIdx.y * chunk;
  const int64_t j_end = min(N, j_begin + chunk);
  int2 u[RI][DP];
  // sums of a tile and of all tiles: chains of 32 terms keep the rounding of a
  // long sum with cancellation at that of its tiles
  T acc[RI][M];
  double tot[RI][M];
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
    for (int c = 0; c < M; ++c) {
      acc[r][c] = A::zero();
      tot[r][c] = 0.0;
    }
  }
  for (int64_t j0 = j_begin; j0 < j_end; j0 += KFIX_TJ) {
    const int jn = (int)min((int64_t)KFIX_TJ, j_end - j0);
    __syncthreads();
    const int4 *src = reinterpret_cast<const int4 *>(uc + j0 * DP);
    for (int i = tid; i < jn * (DP / 2); i += KFIX_THREADS)
      reinterpret_cast<int4 *>(su)[i] = src[i];
    for (int i = tid; i < KFIX_TJ * M; i += KFIX_THREADS) {
      const int c = i / KFIX_TJ, jj = i % KFIX_TJ;
      sv[jj][c] = (jj < jn && c < m) ? A::load(V[(int64_t)c * ldv + j0 + jj]) : A::zero();
    }
    __syncthreads();
#pragma unroll 1
    for (int jj = 0; jj < jn; ++jj) {
      const int4 *v = reinterpret_cast<const int4 *>(su[jj]);
      T kv[RI];
#pragma unroll
      for (int r = 0; r < RI; ++r) kv[r] = fix_kappa<A, KERN, DP>(u[r], v, fs, tab, cst);
#pragma unroll
      for (int c = 0; c < M; ++c)
#pragma unroll
        for (int r = 0; r < RI; ++r) A::fma_(acc[r][c], kv[r], sv[jj][c]);
    }
#pragma unroll
    for (int r = 0; r < RI; ++r)
#pragma unroll
      for (int c = 0; c < M; ++c) {
        tot[r][c] += A::value(acc[r][c]);
        acc[r][c] = A::zero();
      }
  }
  double *out = part + (int64_t)blockIdx.y * M * Nr;
#pragma unroll
  for (int r = 0; r < RI; ++r) {
    const int64_t i = row0 + (int64_t)r * KFIX_THREADS;
    if (i < Nr)
#pragma unroll
      for (int c = 0; c < M; ++c)
        if (c < m) out[(int64_t)c * Nr + i] = tot[r][c];
  }
}

// Symmetric square product: CTA p takes the pair (I, J >= I) of the upper
// triangle of nt tiles of RT points (row-major, ffsym_start) and evaluates its
// entries once for both (K V)_I and (K V)_J; a diagonal pair gives row sums
// only.  Rows 128 at a time, one a thread, against 32 staged columns: the row
// sums stay in registers; a warp's 32 x 32 values pass through shared memory,
// where each lane then takes one column and adds its 32 rows (a store and a
// load an entry against about 5d + 60 instructions to form it again).
// rowpart, colpart[p][c][RT]: the pair's sums.
template <typename A, int KERN, int DP, int M>
__global__ void __launch_bounds__(KFIX_THREADS)
kmvfixsym_kernel(const int2 *__restrict__ u, int64_t N, const FixScale *__restrict__ scale,
                 const double *__restrict__ V, int64_t ldv, int m, int RT, int nt,
                 const ExpFFConsts ec, double *__restrict__ rowpart,
                 double *__restrict__ colpart) {
  using T = typename A::T;
  constexpr int NW = KFIX_THREADS / 32;
  extern __shared__ __align__(16) unsigned char fix_smem[];
  T *scol = reinterpret_cast<T *>(fix_smem);                         // [RT][M]
  T(*sk)[32][33] = reinterpret_cast<T(*)[32][33]>(scol + RT * M);     // [NW]
  __shared__ __align__(16) int2 su[32][DP];
  __shared__ __align__(16) T sv[32][M], svr[KFIX_THREADS][M], sred[NW][32][M];
  __shared__ uint64_t tab[kFixTab];
  __shared__ float cst[KERN == KMATERN && A::kFF ? 68 : 1];
  if (!scale->ok) return;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const FixScale fs = fix_load_scale(scale);
  fix_load_tables<A, KERN>(ec, tab, cst);
  const int64_t p = blockIdx.x;
  const int I = ffsym_row(p, nt);
  const int J = I + (int)(p - ffsym_start(I, nt));
  const bool diag = I == J;
  const int64_t i0 = (int64_t)I * RT, j00 = (int64_t)J * RT;
  for (int i = tid; i < RT * M; i += KFIX_THREADS) scol[i] = A::zero();
  for (int a = 0; a < RT; a += KFIX_THREADS) {
    if (i0 + a >= N) break;
    const int64_t i = i0 + a + tid;
    int2 ui[DP];
    T acc[M];
    double tot[M];
    {
      const int4 *src = reinterpret_cast<const int4 *>(u + min(i, N - 1) * DP);
#pragma unroll
      for (int k = 0; k < DP; k += 2) {
        const int4 q = src[k / 2];
        ui[k] = make_int2(q.x, q.y);
        ui[k + 1] = make_int2(q.z, q.w);
      }
    }
    __syncthreads();
#pragma unroll
    for (int c = 0; c < M; ++c) {
      acc[c] = A::zero();
      tot[c] = 0.0;
      svr[tid][c] = (i < N && c < m) ? A::load(V[(int64_t)c * ldv + i]) : A::zero();
    }
    for (int b = 0; b < RT; b += 32) {
      const int64_t j0 = j00 + b;
      if (j0 >= N) break;
      const int jn = (int)min((int64_t)32, N - j0);
      __syncthreads();
      const int4 *src = reinterpret_cast<const int4 *>(u + j0 * DP);
      for (int e = tid; e < 32 * (DP / 2); e += KFIX_THREADS)
        reinterpret_cast<int4 *>(su)[e] = e < jn * (DP / 2) ? src[e] : make_int4(0, 0, 0, 0);
      for (int e = tid; e < 32 * M; e += KFIX_THREADS) {
        const int c = e >> 5, jj = e & 31;
        sv[jj][c] = (jj < jn && c < m) ? A::load(V[(int64_t)c * ldv + j0 + jj]) : A::zero();
      }
      __syncthreads();
#pragma unroll 2
      for (int jj = 0; jj < 32; ++jj) {
        const T kv = fix_kappa<A, KERN, DP>(ui, reinterpret_cast<const int4 *>(su[jj]), fs, tab, cst);
        if (!diag) sk[warp][jj][lane] = kv;
#pragma unroll
        for (int c = 0; c < M; ++c) A::fma_(acc[c], kv, sv[jj][c]);
      }
#pragma unroll
      for (int c = 0; c < M; ++c) {
        tot[c] += A::value(acc[c]);
        acc[c] = A::zero();
      }
      if (!diag) {
        __syncwarp();
        T cs[M];
#pragma unroll
        for (int c = 0; c < M; ++c) cs[c] = A::zero();
#pragma unroll 2
        for (int r = 0; r < 32; ++r) {
          const T kv = sk[warp][lane][r];
#pragma unroll
          for (int c = 0; c < M; ++c) A::fma_(cs[c], kv, svr[warp * 32 + r][c]);
        }
#pragma unroll
        for (int c = 0; c < M; ++c) sred[warp][lane][c] = cs[c];
        __syncthreads();
        for (int e = tid; e < 32 * M; e += KFIX_THREADS) {
          T t = (&scol[b * M])[e];
#pragma unroll
          for (int w = 0; w < NW; ++w) t = A::add(t, (&sred[w][0][0])[e]);
          (&scol[b * M])[e] = t;
        }
      }
    }
#pragma unroll
    for (int c = 0; c < M; ++c) rowpart[(p * M + c) * RT + a + tid] = tot[c];
  }
  if (diag) return;
  __syncthreads();
  for (int e = tid; e < RT * M; e += KFIX_THREADS)
    colpart[(p * M + e % M) * RT + e / M] = A::value(scol[e]);
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
  const FixScale fs = fix_load_scale(scale);
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
        fix_kappa<FixAccD, KERN, DP>(u, reinterpret_cast<const int4 *>(su[c]), fs, tab, nullptr);
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
  ExpFFConsts ec;
  double *part;
};

struct KmvFixSymArgs {
  const int2 *u;
  int64_t N;
  const FixScale *scale;
  const double *V;
  int64_t ldv;
  int m, RT, nt;
  ExpFFConsts ec;
  double *rowpart, *colpart;
};

// Dynamic shared memory of the symmetric kernel: column sums and the warps'
// values.
inline size_t kmvfixsym_smem(int RT, int M) {
  return (size_t)(RT * M + (KFIX_THREADS / 32) * 32 * 33) * 8;
}

template <typename A, int KERN, int DP>
cudaError_t launch_kmvfix_m(int M, dim3 grid, cudaStream_t s, const KmvFixArgs &a) {
  switch (M) {
#define KRR_CASE(MM)                                                                           \
  case MM:                                                                                     \
    kmvfix_kernel<A, KERN, DP, MM><<<grid, KFIX_THREADS, 0, s>>>(                               \
        a.ur, a.Nr, a.uc, a.scale, a.V, a.ldv, a.N, a.m, a.chunk, a.ec, a.part);                \
    break;
    KRR_CASE(1) KRR_CASE(2) KRR_CASE(4) KRR_CASE(8) KRR_CASE(16)
#undef KRR_CASE
    default:
      return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

template <typename A, int KERN, int DP>
cudaError_t launch_kmvfixsym_m(int M, cudaStream_t s, const KmvFixSymArgs &a) {
  const size_t smem = kmvfixsym_smem(a.RT, M);
  const unsigned grid = (unsigned)(a.nt * (int64_t)(a.nt + 1) / 2);
  switch (M) {
#define KRR_CASE(MM)                                                                            \
  case MM:                                                                                      \
    /* static and dynamic shared memory together pass the default limit */                     \
    if (raise_smem_limit(kmvfixsym_kernel<A, KERN, DP, MM>, smem + 49152) != KRR_OK)             \
      return cudaErrorInvalidValue;                                                             \
    kmvfixsym_kernel<A, KERN, DP, MM><<<grid, KFIX_THREADS, smem, s>>>(                          \
        a.u, a.N, a.scale, a.V, a.ldv, a.m, a.RT, a.nt, a.ec, a.rowpart, a.colpart);             \
    break;
    KRR_CASE(1) KRR_CASE(2) KRR_CASE(4)
#undef KRR_CASE
    default:
      return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

#define KRR_FIX_DP_SWITCH(DP, FN, ...)         \
  switch (DP) {                                \
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

#define KRR_FIX_ACC_SWITCH(DP, FN, ...)           \
  switch (DP) {                                   \
    case 4: return FN<A, KERN, 4>(__VA_ARGS__);   \
    case 8: return FN<A, KERN, 8>(__VA_ARGS__);   \
    case 12: return FN<A, KERN, 12>(__VA_ARGS__); \
    case 16: return FN<A, KERN, 16>(__VA_ARGS__); \
    case 20: return FN<A, KERN, 20>(__VA_ARGS__); \
    case 24: return FN<A, KERN, 24>(__VA_ARGS__); \
    case 28: return FN<A, KERN, 28>(__VA_ARGS__); \
    case 32: return FN<A, KERN, 32>(__VA_ARGS__); \
    default: return cudaErrorInvalidValue;        \
  }

template <typename A, int KERN>
cudaError_t launch_kmvfix(int DP, int M, dim3 grid, cudaStream_t s, const KmvFixArgs &a) {
  KRR_FIX_ACC_SWITCH(DP, launch_kmvfix_m, M, grid, s, a)
}

template <typename A, int KERN>
cudaError_t launch_kmvfixsym(int DP, int M, cudaStream_t s, const KmvFixSymArgs &a) {
  KRR_FIX_ACC_SWITCH(DP, launch_kmvfixsym_m, M, s, a)
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
