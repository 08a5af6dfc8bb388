// Preparation and launch of the fixed-point float64 products (kfix.cuh): the
// range of the points, the common scale, the integer coordinates.
#include <cmath>

#include "kmvfix_kernels.cuh"

namespace krr {

#define KRR_DECL(K)                                                                       \
  cudaError_t launch_kmvfix_##K(int, int, dim3, cudaStream_t, const KmvFixArgs &);          \
  cudaError_t launch_kmvfix_ff_##K(int, int, dim3, cudaStream_t, const KmvFixArgs &);       \
  cudaError_t launch_kmvfixsym_##K(int, int, cudaStream_t, const KmvFixSymArgs &);          \
  cudaError_t launch_kmvfixsym_ff_##K(int, int, cudaStream_t, const KmvFixSymArgs &);
KRR_DECL(gauss)
KRR_DECL(laplace)
KRR_DECL(matern)
#undef KRR_DECL
cudaError_t launch_kfix_columns_gauss(int, const int2 *, int64_t, const FixScale *,
                                      const int64_t *, int, double *, int64_t, cudaStream_t);
cudaError_t launch_kfix_columns_laplace(int, const int2 *, int64_t, const FixScale *,
                                        const int64_t *, int, double *, int64_t, cudaStream_t);
cudaError_t launch_kfix_columns_matern(int, const int2 *, int64_t, const FixScale *,
                                       const int64_t *, int, double *, int64_t, cudaStream_t);

// Block b's smallest and largest value of every coordinate over its share of
// the points: part[b][0 or 1][k].  The active threads of a block are a
// multiple of d, so a thread stays on one coordinate while the block reads
// consecutive memory.  A non-finite value (or one whose range could overflow)
// becomes an infinite range.
constexpr int FIX_RANGE_THREADS = 256;
__global__ void __launch_bounds__(FIX_RANGE_THREADS)
fix_range_kernel(const double *__restrict__ X, int64_t total, int d, int skip,
                 double *__restrict__ part) {
  __shared__ double smin[FIX_RANGE_THREADS], smax[FIX_RANGE_THREADS];
  const int active = FIX_RANGE_THREADS / d * d;
  const int tid = threadIdx.x;
  double lo = INFINITY, hi = -INFINITY;
  if (tid < active) {
    const int64_t step = (int64_t)gridDim.x * active;
    for (int64_t i = (int64_t)blockIdx.x * active + tid; i < total; i += step) {
      const double x = X[i];
      const bool fine = fabs(x) < 1e300;
      lo = fine ? fmin(lo, x) : -INFINITY;
      hi = fine ? fmax(hi, x) : INFINITY;
      if (!fine) break;
    }
  }
  smin[tid] = lo;
  smax[tid] = hi;
  __syncthreads();
  if (tid < d) {
    for (int t = tid + d; t < active; t += d) {
      lo = fmin(lo, smin[t]);
      hi = fmax(hi, smax[t]);
    }
    double *p = part + (int64_t)(skip + blockIdx.x) * 64;
    p[tid] = lo;
    p[32 + tid] = hi;
  }
}

// Centre and fraction bits from the blocks' ranges; one warp.
__global__ void fix_scale_kernel(const double *__restrict__ part, int blocks, int d, int kern,
                                 int ff, double s_hi, double s_lo, FixScale *__restrict__ out) {
  const int k = threadIdx.x;
  double lo = INFINITY, hi = -INFINITY;
  if (k < d)
    for (int b = 0; b < blocks; ++b) {
      lo = fmin(lo, part[(int64_t)b * 64 + k]);
      hi = fmax(hi, part[(int64_t)b * 64 + 32 + k]);
    }
  double ctr = 0.0, half = 0.0;
  if (k < d) {
    ctr = 0.5 * lo + 0.5 * hi;
    half = fmax(hi - ctr, ctr - lo) * s_hi;
    if (!(half < 1e300)) half = INFINITY;   // NaN (infinite ends) included
  }
  out->ctr[k] = ctr;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) half = fmax(half, __shfl_xor_sync(0xffffffffu, half, o));
  if (k != 0) return;
  const int lim[2][3] = {{kFixMaxExpGauss, kFixMaxExpLaplace, kFixMaxExpMatern},
                         {kFixFFMaxExpGauss, kFixFFMaxExpLaplace, kFixFFMaxExpMatern}};
  const int e_max = lim[ff][kern];
  // 2^e above the half-range with room for the coordinate rounding
  int e = kFixMinExp;
  while (e <= e_max && half * (1.0 + 0x1p-26) >= ldexp(1.0, e)) ++e;
  out->ok = e <= e_max ? 1 : 0;
  e = min(e, e_max);
  out->s_hi = s_hi;
  out->s_lo = s_lo;
  out->s1_max = 0;
  out->r2_scale = 0.0;
  out->bias = 0;
  out->s1_near = 0;
  if (kern == KLAPLACE) {
    out->limb = 0;
    out->q = (ff ? kFixFFL1Bits : kFixL1Bits) - e;
    out->r = out->q - 54;
    return;
  }
  out->limb = ff ? kFixFFLimb : kFixLimb;
  out->q = (ff ? 53 : 57) - e;
  out->r = (ff ? 26 : 30) - 2 * e;
  const int left = (ff ? 24 : 28) - out->r;   // left shift of S1 to 54 fraction bits
  out->r2_scale = ldexp(1.0, 30 - 2 * out->q);
  // (without a shift every sum of squares stays below E = 512)
  out->s1_max = left == 0 ? INT64_MAX : (int64_t)((1022ull << 54) >> left);
  if (ff) {
    // the mean of a squared difference of low limbs uniform over 2^25 values is
    // 2^50 / 6 a coordinate (padded coordinates have none); 2^50 S1 is worth
    // 2^(2 e - 56) S1
    out->bias = (int64_t)d * (1 << 24) / 6;
    out->s1_near = 1u << (56 - 2 * e - kFixNearExp - 32);
  }
}

__global__ void fix_convert_kernel(const double *__restrict__ X, int64_t N, int d, int dp,
                                   const FixScale *__restrict__ scale, int2 *__restrict__ u) {
  if (!scale->ok) return;
  const double s_hi = scale->s_hi, s_lo = scale->s_lo;
  const int q = scale->q, limb = scale->limb;
  const int64_t total = N * dp;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = e / dp;
    const int k = (int)(e - i * dp);
    int2 v = make_int2(0, 0);
    if (k < d) {
      const int64_t c = fix_coord(X[i * d + k], scale->ctr[k], s_hi, s_lo, q);
      if (limb == 0) {
        v = make_int2((int)(uint32_t)(uint64_t)c, (int)(c >> 32));
      } else {
        fix_limbs(c, limb, &v.x, &v.y);
      }
    }
    u[e] = v;
  }
}

krr_status fix_scale(const double *A, int64_t na, const double *B, int64_t nb, int d, int kern,
                     double sigma, bool ff, cudaStream_t s, DevBuf<FixScale> &out) {
  KRR_REQUIRE(d >= 1 && d <= 32, "d must be in [1, 32]");
  // sqrt(log2 e / 2), log2 e and sqrt(5) as unevaluated sums, divided by sigma
  static const double num[3][2] = {{0x1.b2da4e9808a53p-1, -0x1.dede1a6b5e413p-56},
                                   {0x1.71547652b82fep+0, 0x1.777d0ffda0d24p-56},
                                   {0x1.1e3779b97f4a8p+1, -0x1.f506319fcfd19p-54}};
  const double s_hi = num[kern][0] / sigma;
  const double s_lo = (std::fma(-s_hi, sigma, num[kern][0]) + num[kern][1]) / sigma;
  // about 2048 values a block: few blocks for the scale kernel's serial loop
  auto blocks = [&](int64_t n) {
    const int64_t g = (n * d + 2047) / 2048;
    return (int)std::min<int64_t>(std::max<int64_t>(g, 1), 2 * num_sms());
  };
  const int ga = blocks(na), gb = B ? blocks(nb) : 0;
  DevBuf<double> part;
  KRR_TRY(part.alloc((size_t)(ga + gb) * 64, s));
  KRR_TRY(out.alloc(1, s));
  fix_range_kernel<<<ga, FIX_RANGE_THREADS, 0, s>>>(A, na * d, d, 0, part.p);
  KRR_LAUNCH_CHECK();
  if (B) {
    fix_range_kernel<<<gb, FIX_RANGE_THREADS, 0, s>>>(B, nb * d, d, ga, part.p);
    KRR_LAUNCH_CHECK();
  }
  fix_scale_kernel<<<1, 32, 0, s>>>(part.p, ga + gb, d, kern, ff ? 1 : 0, s_hi, s_lo, out.p);
  KRR_LAUNCH_CHECK();
  return KRR_OK;
}

krr_status fix_points(const double *Xd, int64_t N, int d, const FixScale *scale, cudaStream_t s,
                      DevBuf<int2> &u) {
  const int dp = (d + 3) / 4 * 4;
  KRR_TRY(u.alloc((size_t)N * dp, s));
  const int64_t g = std::min<int64_t>((N * dp + 255) / 256, (int64_t)num_sms() * 16);
  fix_convert_kernel<<<(unsigned)g, 256, 0, s>>>(Xd, N, d, dp, scale, u.p);
  KRR_LAUNCH_CHECK();
  return KRR_OK;
}

krr_status prepare_points_f64(const double *Xd, int64_t N, int d, int kern, double sigma,
                              cudaStream_t s, PointsF64 &P, bool wait) {
  P.X = Xd;
  P.N = N;
  P.d = d;
  P.kern = kern;
  P.sigma = sigma;
  P.known = -1;
  KRR_TRY(fix_scale(Xd, N, nullptr, 0, d, kern, sigma, false, s, P.scale));
  KRR_TRY(fix_points(Xd, N, d, P.scale.p, s, P.u));
  if (wait) {
    int ok = 0;
    KRR_CUDA_TRY(cudaMemcpyAsync(&ok, &P.scale.p->ok, sizeof(int), cudaMemcpyDeviceToHost, s));
    KRR_CUDA_TRY(cudaStreamSynchronize(s));
    P.known = ok;
  }
  return KRR_OK;
}

cudaError_t launch_kmvfix_any(int kern, bool ff, int DP, int M, dim3 g, cudaStream_t s,
                              const KmvFixArgs &a) {
  switch (kern) {
    case KGAUSS: return ff ? launch_kmvfix_ff_gauss(DP, M, g, s, a) : launch_kmvfix_gauss(DP, M, g, s, a);
    case KLAPLACE:
      return ff ? launch_kmvfix_ff_laplace(DP, M, g, s, a) : launch_kmvfix_laplace(DP, M, g, s, a);
    case KMATERN:
      return ff ? launch_kmvfix_ff_matern(DP, M, g, s, a) : launch_kmvfix_matern(DP, M, g, s, a);
  }
  return cudaErrorInvalidValue;
}

cudaError_t launch_kmvfixsym_any(int kern, bool ff, int DP, int M, cudaStream_t s,
                                 const KmvFixSymArgs &a) {
  switch (kern) {
    case KGAUSS: return ff ? launch_kmvfixsym_ff_gauss(DP, M, s, a) : launch_kmvfixsym_gauss(DP, M, s, a);
    case KLAPLACE:
      return ff ? launch_kmvfixsym_ff_laplace(DP, M, s, a) : launch_kmvfixsym_laplace(DP, M, s, a);
    case KMATERN:
      return ff ? launch_kmvfixsym_ff_matern(DP, M, s, a) : launch_kmvfixsym_matern(DP, M, s, a);
  }
  return cudaErrorInvalidValue;
}

krr_status kfix_columns(const PointsF64 &P, const int64_t *cols, int nc, double *G, int64_t ldg,
                        cudaStream_t s) {
  const int DP = (P.d + 3) / 4 * 4;
  cudaError_t e = cudaErrorInvalidValue;
  switch (P.kern) {
    case KGAUSS:
      e = launch_kfix_columns_gauss(DP, P.u.p, P.N, P.scale.p, cols, nc, G, ldg, s);
      break;
    case KLAPLACE:
      e = launch_kfix_columns_laplace(DP, P.u.p, P.N, P.scale.p, cols, nc, G, ldg, s);
      break;
    case KMATERN:
      e = launch_kfix_columns_matern(DP, P.u.p, P.N, P.scale.p, cols, nc, G, ldg, s);
      break;
  }
  count_launch();
  if (e != cudaSuccess) {
    set_error("kernel column launch failed: %s", cudaGetErrorString(e));
    return KRR_ECUDA;
  }
  return KRR_OK;
}

}  // namespace krr
