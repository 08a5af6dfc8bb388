// Host side of the tcgen05 product (kmvtc5_kernels.cuh): the split operands
// and their TMA tensor maps, the launch over right-hand-side groups of at
// most 16, and the reduction of the per-CTA segment partial sums.
#include <cuda_fp16.h>
#include <cudaTypedefs.h>

#include <algorithm>
#include <atomic>
#include <map>
#include <mutex>
#include <tuple>

#include "kmv.cuh"
#include "kmvtc5_kernels.cuh"

namespace krr {

// ------------------------------------------------------------ preparation
// One thread per point: centred, scaled coordinates split as h + l, c split
// as c1 + c2 + c3; writes the row operand xa and the column operand xb
// (kb = 2 nh + csep blocks of 16 halves each, stored K-block-major: block q
// of point i at (q N + i) 16).  A coordinate or c outside the split's range
// sets *bad.  xa or xb may be NULL (a rectangular product needs one of them).
// cshift is added to c on both sides (7 for the Gaussian: D = log2 kappa + 14).
// A block of 16 halves is assembled in registers and stored as two 16-byte
// words, and what follows the difference and the scaling, which are float64
// (at 1.9 operations a clock and SM they bound the kernel), is float32.
template <int NH, int CSEP>
__global__ void __launch_bounds__(128)
prepare_tc5_kernel(const double *__restrict__ X, int64_t N, int d,
                   const double *__restrict__ mean, double scale, double cshift,
                   uint4 *__restrict__ xa, uint4 *__restrict__ xb, int *__restrict__ bad) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= N) return;
  auto store = [&](uint4 *base, int q, const uint32_t (&w)[8]) {
    if (!base) return;
    uint4 *dst = base + ((int64_t)q * N + i) * 2;
    dst[0] = make_uint4(w[0], w[1], w[2], w[3]);
    dst[1] = make_uint4(w[4], w[5], w[6], w[7]);
  };
  auto pack = [](__half lo, __half hi) {
    return (uint32_t)__half_as_ushort(lo) | ((uint32_t)__half_as_ushort(hi) << 16);
  };
  // |h + l|^2 as an unevaluated float sum: the three products of a square are
  // exact in float32 (h and l have 11 bits)
  float sh = 0.0f, sl = 0.0f;
  auto add = [&](float v) {
    const float t = __fadd_rn(sh, v), z = __fsub_rn(t, sh);
    sl = __fadd_rn(sl, __fadd_rn(__fsub_rn(sh, __fsub_rn(t, z)), __fsub_rn(v, z)));
    sh = t;
  };
  bool out_of_range = false;
  uint32_t hw[8];
#pragma unroll
  for (int b = 0; b < NH; ++b) {
    uint32_t lw[8];
#pragma unroll
    for (int t = 0; t < 8; ++t) {
      __half h[2] = {__ushort_as_half(0), __ushort_as_half(0)}, l[2] = {h[0], h[0]};
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const int k = b * 16 + 2 * t + u;
        if (k < d) {
          const double v = (X[i * d + k] - mean[k]) * scale;
          const float vh = (float)v, vl = (float)(v - (double)vh);
          if (!(fabsf(vh) <= T5_MAX_COORD)) out_of_range = true;
          h[u] = __float2half_rn(vh);
          const float hf = __half2float(h[u]);
          l[u] = __float2half_rn(__fadd_rn(__fsub_rn(vh, hf), vl));
          const float lf = __half2float(l[u]);
          add(__fmul_rn(hf, hf));
          add(__fmul_rn(2.0f * hf, lf));
          sl = __fmaf_rn(lf, lf, sl);
        }
      }
      hw[t] = pack(h[0], h[1]);
      lw[t] = pack(l[0], l[1]);
    }
    store(xa, NH + b, lw);
    store(xb, NH + b, lw);
    if (b + 1 < NH || CSEP) {
      store(xa, b, hw);
      store(xb, b, hw);
    }
  }
  const double c = -0.5 * ((double)sh + (double)sl) + cshift;
  if (!(fabs(c) <= (double)T5_MAX_C)) out_of_range = true;
  const __half c1 = __double2half(c);
  const double r1 = c - (double)__half2float(c1);
  const __half c2 = __double2half(r1);
  const __half c3 = __double2half(r1 - (double)__half2float(c2));
  const __half one = __double2half(1.0), zero = __double2half(0.0);
  // c-part: its own block, or positions 10..15 of the last H block (those
  // coordinates are beyond d, so their H and L entries are zero); the row
  // operand holds (c1, c2, c3, 1, 1, 1), the column operand (1, 1, 1, c1, c2, c3)
  const uint32_t pa[3] = {pack(c1, c2), pack(c3, one), pack(one, one)};
  const uint32_t pb[3] = {pack(one, one), pack(one, c1), pack(c2, c3)};
  if (CSEP) {
    const uint32_t z = pack(zero, zero);
    const uint32_t wa[8] = {pa[0], pa[1], pa[2], z, z, z, z, z};
    const uint32_t wb[8] = {pb[0], pb[1], pb[2], z, z, z, z, z};
    store(xa, 2 * NH, wa);
    store(xb, 2 * NH, wb);
  } else {
    const uint32_t wa[8] = {hw[0], hw[1], hw[2], hw[3], hw[4], pa[0], pa[1], pa[2]};
    const uint32_t wb[8] = {hw[0], hw[1], hw[2], hw[3], hw[4], pb[0], pb[1], pb[2]};
    store(xa, NH - 1, wa);
    store(xb, NH - 1, wb);
  }
  if (out_of_range) *bad = 1;
}

static PFN_cuTensorMapEncodeTiled_v12000 tensormap_encoder() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void *p = nullptr;
    cudaDriverEntryPointQueryResult q = cudaDriverEntryPointSymbolNotFound;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault,
                                         &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = (PFN_cuTensorMapEncodeTiled_v12000)p;
    else
      cudaGetLastError();
  });
  return fn;
}

// 3-D map over a kb x N x 16 fp16 operand (K-block-major): boxes of 16 halves
// (one K-block row, 32 bytes) x 128 points x kb blocks, 32-byte swizzle, zero
// fill beyond N.  Each block of a box is a contiguous 4 KB range.
static krr_status encode_operand_map(CUtensorMap *map, const uint16_t *ptr, int64_t N, int kb) {
  auto enc = tensormap_encoder();
  if (!enc) {
    set_error("cuTensorMapEncodeTiled is not available from the driver");
    return KRR_ECUDA;
  }
  const cuuint64_t dims[3] = {16, (cuuint64_t)N, (cuuint64_t)kb};
  const cuuint64_t strides[2] = {32, (cuuint64_t)N * 32};
  const cuuint32_t box[3] = {16, (cuuint32_t)T5_TM, (cuuint32_t)kb};
  const cuuint32_t estr[3] = {1, 1, 1};
  const CUresult r = enc(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 3, (void *)ptr, dims, strides, box,
                         estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_32B,
                         CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) {
    set_error("cuTensorMapEncodeTiled failed (%d)", (int)r);
    return KRR_ECUDA;
  }
  return KRR_OK;
}

// Allocates and fills P's tcgen05 operands and encodes their maps (P.nh5 >
// 0); a point outside the split's range sets *bad_dev (cleared by the
// caller).  rows, cols: which operands are wanted.
static krr_status tc5_operands(const double *Xd, cudaStream_t s, PointsF32 &P, const double *mean,
                               bool rows, bool cols, int *bad_dev) {
  const int nh = t5_nh(P.d), csep = t5_csep(P.d), kb = t5_kb(nh, csep);
  const double log2e = 1.4426950408889634;
  const double scale = (P.kern == KGAUSS) ? std::sqrt(log2e) / P.sigma : std::sqrt(5.0) / P.sigma;
  if (rows) KRR_TRY(P.xa5.alloc((size_t)P.N * kb * 16, s));
  if (cols) KRR_TRY(P.xb5.alloc((size_t)P.N * kb * 16, s));
  uint4 *xa = reinterpret_cast<uint4 *>(rows ? P.xa5.p : nullptr);
  uint4 *xb = reinterpret_cast<uint4 *>(cols ? P.xb5.p : nullptr);
  const double cshift = P.kern == KGAUSS ? 7.0 : 0.0;
  const unsigned grid = ceil_div(P.N, 128);
#define KRR_PREP(NH, CS)                                                                     \
  if (nh == NH && csep == CS)                                                                \
  prepare_tc5_kernel<NH, CS><<<grid, 128, 0, s>>>(Xd, P.N, P.d, mean, scale, cshift, xa, xb, \
                                                  bad_dev)
  KRR_PREP(1, 0);
  KRR_PREP(1, 1);
  KRR_PREP(2, 0);
  KRR_PREP(2, 1);
#undef KRR_PREP
  KRR_LAUNCH_CHECK();
  if (rows) KRR_TRY(encode_operand_map(&P.ma5, P.xa5.p, P.N, kb));
  if (cols) KRR_TRY(encode_operand_map(&P.mb5, P.xb5.p, P.N, kb));
  P.nh5 = nh;
  P.csep5 = csep;
  return KRR_OK;
}

// Builds P's tcgen05 operands (P.nh5 > 0 on success; left at 0 when a point is
// outside the split's range) with the centre mean_dev, or P.mean.
krr_status prepare_points_tc5(const double *Xd, cudaStream_t s, PointsF32 &P, int *h_bad_out,
                              const double *mean_dev) {
  P.nh5 = 0;
  *h_bad_out = 0;
  if (P.kern == KLAPLACE || P.d > 32 || P.N == 0) return KRR_OK;
  DevBuf<int> bad;
  KRR_TRY(bad.alloc(1, s));
  KRR_CUDA_TRY(cudaMemsetAsync(bad.p, 0, sizeof(int), s));
  KRR_TRY(tc5_operands(Xd, s, P, mean_dev ? mean_dev : P.mean.p, true, true, bad.p));
  int h_bad = 0;
  KRR_CUDA_TRY(cudaMemcpyAsync(&h_bad, bad.p, sizeof(int), cudaMemcpyDeviceToHost, s));
  KRR_CUDA_TRY(cudaStreamSynchronize(s));
  if (h_bad) {
    P.nh5 = 0;
    P.xa5.release();
    P.xb5.release();
    *h_bad_out = 1;
  }
  return KRR_OK;
}

// --------------------------------------------------------------- faults
// Set by a CTA whose bounded wait gave up (one flag per device, read and
// cleared by tc5_check_fault).
__device__ int g_t5_fault;

int *tc5_fault_ptr() {
  static std::mutex mtx;
  static int *ptrs[64] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return nullptr;
  std::lock_guard<std::mutex> lk(mtx);
  if (!ptrs[dev]) {
    void *p = nullptr;
    if (cudaGetSymbolAddress(&p, g_t5_fault) != cudaSuccess) {
      cudaGetLastError();
      return nullptr;
    }
    ptrs[dev] = static_cast<int *>(p);
  }
  return ptrs[dev];
}

krr_status tc5_check_fault(cudaStream_t s) {
  int *f = tc5_fault_ptr();
  if (!f) return KRR_OK;
  int h = 0;
  KRR_CUDA_TRY(cudaMemcpyAsync(&h, f, sizeof(int), cudaMemcpyDeviceToHost, s));
  KRR_CUDA_TRY(cudaStreamSynchronize(s));
  if (h) {
    KRR_CUDA_TRY(cudaMemsetAsync(f, 0, sizeof(int), s));
    set_error("a bounded wait of the tensor-core product gave up (device-side timeout)");
    return KRR_ETIMEOUT;
  }
  return KRR_OK;
}

// Diagnostic of the bounded waits: one thread waits on an mbarrier that no
// arrival ever completes, for `budget` SM clock cycles, with the routine the
// product's roles use, then takes the timeout path (the fault flag).
__global__ void t5_wait_selftest_kernel(int *fault, long long budget) {
  __shared__ __align__(8) uint64_t bar;
  __shared__ int abort_flag;
  if (threadIdx.x != 0) return;
  const uint32_t b = bw::smem_u32(&bar);
  bw::mbar_init(b, 1);
  abort_flag = 0;
  bw::fence_mbar_init();
  if (!bw::mbar_wait_abortable(b, 0, budget, &abort_flag)) atomicOr(fault, 1);
}

krr_status tc5_wait_selftest(long long budget, cudaStream_t s) {
  KRR_REQUIRE(budget >= 0 && budget <= (1LL << 31), "wait budget: 0 to 2^31 cycles");
  int *f = tc5_fault_ptr();
  KRR_REQUIRE(f != nullptr, "no fault flag on this device");
  t5_wait_selftest_kernel<<<1, 32, 0, s>>>(f, budget);
  KRR_LAUNCH_CHECK();
  return tc5_check_fault(s);
}

// ------------------------------------------------------------ reduction
// Y[c][i] = sum of the partial sums of row i over the CTAs covering its row
// block (CTA order) and column groups, + lambda V[c][i] when V is given.  With
// vexp (TV variants) the partial sums of right-hand side c carry the factor
// 2^(14 + vexp[c]), which is divided out in float64.
// TV5: the type of V and Y.  flags (optional): {a point outside the split's
// range (nothing was summed then), a bounded wait gave up}, for one read-back
// after the product.
template <typename TV5>
__global__ void t5_reduce_kernel(const float *__restrict__ part, int64_t Nr, int m, int M, int C,
                                 int64_t T, int G, int J, int CG, const int *__restrict__ vexp,
                                 double lambda, const TV5 *__restrict__ V, int64_t ldv,
                                 TV5 *__restrict__ Y, int64_t ldy, const int *__restrict__ fault,
                                 int *__restrict__ flags) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (flags && i == 0) flags[1] = *fault;
  if (i >= Nr || (flags && flags[0])) return;
  const int64_t rb = i / T5_RB;
  const int r = (int)(i % T5_RB);
  const int b_lo = t5_cta_of(rb * C, T, G);
  const int b_hi = t5_cta_of(rb * C + C - 1, T, G);
  for (int c = 0; c < m; ++c) {
    double acc = 0.0;   // a row block's segments may come from many CTAs
    for (int b = b_lo; b <= b_hi; ++b) {
      const int64_t j = rb - ((int64_t)b * T / G) / C;
      for (int cg = 0; cg < CG; ++cg)
        acc += (double)part[((((int64_t)b * J + j) * CG + cg) * M + c) * T5_RB + r];
    }
    if (vexp) acc = ldexp(acc, -14 - vexp[c]);
    Y[(int64_t)c * ldy + i] =
        V ? (TV5)(acc + lambda * (double)V[(int64_t)c * ldv + i]) : (TV5)acc;
  }
}

// The same sums for row blocks that many CTAs share (few rows against many
// columns, or a small product): 32 rows a block, whose eight warps take every
// eighth segment each; the warps' sums are added in warp order.  With one
// thread a row the chain of loads took 13.3 us at N = 2000 (32 segments a row)
// and 16.2 us at 1000 rows by 2e5 columns (78).
constexpr int T5_RED_WARPS = 8;
template <typename TV5>
__global__ void __launch_bounds__(32 * T5_RED_WARPS)
t5_reduce_many_kernel(const float *__restrict__ part, int64_t Nr, int m, int M, int C, int64_t T,
                      int G, int J, int CG, const int *__restrict__ vexp, double lambda,
                      const TV5 *__restrict__ V, int64_t ldv, TV5 *__restrict__ Y, int64_t ldy,
                      const int *__restrict__ fault, int *__restrict__ flags) {
  __shared__ double red[T5_RED_WARPS][32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t i0 = (int64_t)blockIdx.x * 32, i = i0 + lane;
  const int c = blockIdx.y;
  if (flags && i0 == 0 && c == 0 && threadIdx.x == 0) flags[1] = *fault;
  if (flags && flags[0]) return;
  const int64_t rb = i0 / T5_RB;
  const int r = (int)(i0 % T5_RB) + lane;
  const int b_lo = t5_cta_of(rb * C, T, G);
  const int b_hi = t5_cta_of(rb * C + C - 1, T, G);
  double acc = 0.0;
  for (int b = b_lo + warp; b <= b_hi; b += T5_RED_WARPS) {
    const int64_t j = rb - ((int64_t)b * T / G) / C;
    for (int cg = 0; cg < CG; ++cg)
      acc += (double)part[((((int64_t)b * J + j) * CG + cg) * M + c) * T5_RB + r];
  }
  red[warp][lane] = acc;
  __syncthreads();
  if (warp != 0 || i >= Nr) return;
#pragma unroll
  for (int w = 1; w < T5_RED_WARPS; ++w) acc += red[w][lane];
  if (vexp) acc = ldexp(acc, -14 - vexp[c]);
  Y[(int64_t)c * ldy + i] =
      V ? (TV5)(acc + lambda * (double)V[(int64_t)c * ldv + i]) : (TV5)acc;
}

// Right-hand sides of the column points as the kernel's shared tiles hold
// them: for column tile t (of TN points), pair cp of right-hand sides and pair
// jp of columns, {v_2cp(j), v_2cp(j + 1), v_2cp+1(j), v_2cp+1(j + 1)}, j = t TN
// + 2 jp, times vscale (zero beyond Nc or m); vscale = 2^-14 for the Gaussian,
// whose kernel values come scaled by 2^14.
template <typename TV5>
__global__ void t5_vpair_kernel(const TV5 *__restrict__ V, int64_t ldv, int64_t Nc, int m,
                                int MP, int C, int TN, float vscale, float4 *__restrict__ vpair) {
  const int TN2 = TN / 2;
  const int64_t total = (int64_t)C * MP * TN2;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int c = 2 * (int)((e / TN2) % MP);
    const int64_t j = e / ((int64_t)TN2 * MP) * TN + 2 * (e % TN2);
    auto val = [&](int cc, int64_t jj) {
      return cc < m && jj < Nc ? (float)V[(int64_t)cc * ldv + jj] * vscale : 0.0f;
    };
    vpair[e] = make_float4(val(c, j), val(c, j + 1), val(c + 1, j), val(c + 1, j + 1));
  }
}

// Largest |v| of each right-hand side (m <= 16) over this block's grid-stride
// share of the Nc points: bmax[block][c].
constexpr int T5_VMAX_BLOCKS = 256;
constexpr int T5_MAX_M = 16;   // right-hand sides of one launch
template <typename TV5>
__global__ void t5_vmax_kernel(const TV5 *__restrict__ V, int64_t ldv, int64_t Nc, int m,
                               float *__restrict__ bmax) {
  __shared__ float red[8][T5_MAX_M];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int c = 0; c < T5_MAX_M; ++c) {
    float mx = 0.0f;
    if (c < m)
      for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < Nc;
           j += (int64_t)gridDim.x * blockDim.x)
        mx = fmaxf(mx, fabsf((float)V[(int64_t)c * ldv + j]));
    for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
    if (lane == 0) red[warp][c] = mx;
  }
  __syncthreads();
  if (threadIdx.x < T5_MAX_M) {
    float mx = 0.0f;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) mx = fmaxf(mx, red[w][threadIdx.x]);
    bmax[blockIdx.x * T5_MAX_M + threadIdx.x] = mx;
  }
}

__device__ __forceinline__ uint32_t t5_pack_halves(__half lo, __half hi) {
  return (uint32_t)__half_as_ushort(lo) | ((uint32_t)__half_as_ushort(hi) << 16);
}

// Right-hand sides as mma.sync B fragments for the TV variants.  Column c is
// scaled by s_c = 2^vexp[c], the power of two that brings its largest |v|
// into [2^13, 2^14), and split into fp16 halves v s_c = v_hi + v_lo.  B slot n
// of fragment f: v_hi of column n (n < M) and v_lo of column n - M (M <= n <
// 2M) for M <= 4; for M = 8 and 16, v_hi (f < M / 8) or v_lo of column n + 8
// (f mod M / 8).  For
// column tile t, batch bt of 16 columns, fragment f and lane 4 g + q, frag
// holds {B(2q, g), B(2q + 1, g)}, {B(2q + 8, g), B(2q + 9, g)} over the
// batch's columns (zero beyond Nc, m or 2M).  Every block derives the scales
// from bmax (gmax blocks); block 0 also stores vexp for the reduction.
template <typename TV5>
__global__ void t5_vfrag_kernel(const TV5 *__restrict__ V, int64_t ldv, int64_t Nc, int m,
                                int M, int C, int TN, const float *__restrict__ bmax, int gmax,
                                uint2 *__restrict__ frag, int *__restrict__ vexp) {
  __shared__ float sc[T5_MAX_M];
  if (threadIdx.x < T5_MAX_M) {
    float mx = 0.0f;
    for (int q = 0; q < gmax; ++q) mx = fmaxf(mx, bmax[q * T5_MAX_M + threadIdx.x]);
    int e = 0;
    if (mx > 0.0f && mx <= 3.4028234663852886e38f) {
      int E = 0;
      frexpf(mx, &E);   // mx < 2^E
      e = min(max(14 - E, -126), 126);
    }
    sc[threadIdx.x] = ldexpf(1.0f, e);
    if (blockIdx.x == 0) vexp[threadIdx.x] = e;
  }
  __syncthreads();
  const int NB = t5_nfrag(M);
  const int nbat = TN / 16;
  const int64_t total = (int64_t)C * nbat * NB * 32;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int lane = (int)(e % 32);
    const int f = (int)((e / 32) % NB);
    const int bt = (int)((e / (32 * NB)) % nbat);
    const int64_t t = e / ((int64_t)32 * NB * nbat);
    const int g = lane >> 2, q = lane & 3;
    int c = g + 8 * (NB > 1 ? f % (NB / 2) : 0);
    bool lo = 2 * f >= NB, live = true;
    if (NB == 1) {
      lo = g >= M;
      c = lo ? g - M : g;
      live = g < 2 * M;
    }
    const int64_t j0 = t * TN + bt * 16;
    auto slot = [&](int k) -> __half {
      const int64_t j = j0 + k;
      if (!live || c >= m || j >= Nc) return __float2half_rn(0.0f);
      const float vs = (float)V[(int64_t)c * ldv + j] * sc[c];
      const __half h = __float2half_rn(vs);
      return lo ? __float2half_rn(vs - __half2float(h)) : h;
    };
    frag[e] = make_uint2(t5_pack_halves(slot(2 * q), slot(2 * q + 1)),
                         t5_pack_halves(slot(2 * q + 8), slot(2 * q + 9)));
  }
}

// ----------------------------------------------------------- variants
// Epilogue variant of the product: forced process-wide (1..T5_NVARIANTS), or
// 0: chosen per shape by timing every valid variant on the caller's stream at
// the first product of that shape while autotuning is on, else the default.
// Results of different variants differ only in the summation order of the
// column groups (rounding level).
static_assert(T5_NVARIANTS == KRR_PRODUCT_VARIANTS, "variant count of the ABI");
// Untuned default.  Square products of 5 and more right-hand sides take the
// tensor-core sums (9): 2.93 ms against 3.59 ms at N = 1e5, d = 16, m = 8.
// Below, the FMA sums, with 8 warps (3) where they are bound by the FMA pipe
// (Gaussian, 3 or 4 right-hand sides, d <= 16: 2.15 ms against 2.25 ms with
// 16) and with 16 (2) otherwise: 1.61 against 1.98 ms for m = 2, 2.43 against
// 2.60 for d = 30, 4.35 against 5.15 for Matern.
static int t5_default_variant(const PointsF32 &P, int M, bool square) {
  if (M >= 8) return square ? 9 : 3;
  return P.kern == KGAUSS && M == 4 && P.nh5 == 1 ? 3 : 2;
}
static std::atomic<int> g_t5_variant{0};
static std::mutex g_t5_mtx;
struct T5Tune {
  int best = 0;
  float ms[T5_NVARIANTS + 1] = {};
};
static std::map<std::tuple<int, int, int, int, int64_t, int64_t, bool>, T5Tune> g_t5_tuned;

krr_status set_tc5_variant(int v) {
  KRR_REQUIRE(v >= 0 && v <= T5_NVARIANTS, "unknown product variant %d", v);
  g_t5_variant.store(v);
  return KRR_OK;
}

bool tc5_tuned(int kern, int d, int M, int64_t N, int *best, float *ms) {
  const int nh = t5_nh(d), csep = t5_csep(d);
  std::lock_guard<std::mutex> lk(g_t5_mtx);
  auto it = g_t5_tuned.find(std::make_tuple(kern, nh, csep, M, N, N, true));
  if (it == g_t5_tuned.end()) return false;
  *best = it->second.best;
  if (ms)
    for (int v = 1; v <= T5_NVARIANTS; ++v) ms[v - 1] = it->second.ms[v];
  return true;
}

// ------------------------------------------------------------------ launch
// Work geometry of one variant: column tiles of TN points, pairs (row block,
// column tile), grid and segments per CTA.
struct T5Geometry {
  int TN = 128, C = 0, G = 0, J = 1;
  int64_t T = 0;
};

static T5Geometry t5_geometry(int64_t Nr, int64_t Nc, int TN) {
  T5Geometry g;
  g.TN = TN;
  const int64_t Rb = (Nr + T5_RB - 1) / T5_RB;
  g.C = (int)((Nc + TN - 1) / TN);
  g.T = Rb * g.C;
  g.G = (int)std::min<int64_t>(num_sms(), g.T);
  for (int b = 0; b < g.G; ++b) {
    const int64_t p0 = (int64_t)b * g.T / g.G, p1 = (int64_t)(b + 1) * g.T / g.G;
    g.J = std::max<int>(g.J, (int)((p1 - 1) / g.C - p0 / g.C + 1));
  }
  return g;
}

// Scratch of one launch: partial sums (room for 4 column groups), the
// right-hand-side quadruples or B fragments (16-byte aligned), the block
// maxima of V and the scale exponents (TV variants).
static size_t t5_npart(const T5Geometry &g, int M) { return (size_t)g.G * g.J * 4 * M * T5_RB; }
static size_t t5_nrhs(const T5Geometry &g, int M) {
  return (size_t)g.C * g.TN * t5_vstage(M) / (4 * 128);   // floats of a column tile's stage
}
static size_t t5_scratch_floats(const T5Geometry &g, int M) {
  return t5_npart(g, M) + t5_nrhs(g, M) + (T5_VMAX_BLOCKS + 1) * T5_MAX_M;
}
static int *t5_vexp(float *part, const T5Geometry &g, int M) {
  return reinterpret_cast<int *>(part + t5_npart(g, M) + t5_nrhs(g, M) + T5_VMAX_BLOCKS * T5_MAX_M);
}

// Stages V for this geometry and launches the product; returns the launch's
// error.  part must hold t5_scratch_floats(g, M) floats.  skip: see T5Args (NULL
// while tuning, whose times would be those of an empty kernel).
template <typename TV5>
static cudaError_t t5_launch(const PointsF32 &R, const PointsF32 &P, int M, int variant,
                             const T5Geometry &g, const TV5 *Vg, int64_t ldv, int mg,
                             float *part, int *fault, const int *skip, cudaStream_t s,
                             bool timed) {
  float *vbuf = part + t5_npart(g, M);
  cudaError_t e = cudaSuccess;
  if (t5_variant_tv(variant)) {
    float *bmax = vbuf + t5_nrhs(g, M);
    const int gmax = (int)std::min<int64_t>((P.N + 255) / 256, T5_VMAX_BLOCKS);
    t5_vmax_kernel<<<gmax, 256, 0, s>>>(Vg, ldv, P.N, mg, bmax);
    count_launch();
    const int NB = t5_nfrag(M);
    const int64_t total = (int64_t)g.C * (g.TN / 16) * NB * 32;
    const int blocks = (int)std::min<int64_t>((total + 255) / 256, 4096);
    t5_vfrag_kernel<<<blocks, 256, 0, s>>>(Vg, ldv, P.N, mg, M, g.C, g.TN, bmax, gmax,
                                           reinterpret_cast<uint2 *>(vbuf), t5_vexp(part, g, M));
    count_launch();
  } else {
    const int64_t total = (int64_t)g.C * (M / 2) * (g.TN / 2);
    const int blocks = (int)std::min<int64_t>((total + 255) / 256, 4096);
    t5_vpair_kernel<<<blocks, 256, 0, s>>>(Vg, ldv, P.N, mg, M / 2, g.C, g.TN,
                                           P.kern == KGAUSS ? 0x1p-14f : 1.0f,
                                           reinterpret_cast<float4 *>(vbuf));
    count_launch();
  }
  e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  const T5Args args{reinterpret_cast<const float4 *>(vbuf), P.N, part, g.C, g.T, g.J, fault, skip};
  const int nh = P.nh5, csep = P.csep5, kb = t5_kb(nh, csep);
  // at least half of an SM's shared memory: one CTA per SM (each takes all
  // 512 TMEM columns)
  const int ew = t5_variant_ew(variant);
  const size_t smem = std::max<size_t>(
      t5_smem_bytes(kb, M, t5_tot_floats(ew, M, t5_variant_tv(variant))),
      116 * 1024);
  const bool tv = t5_variant_tv(variant), gauss = P.kern == KGAUSS;
  KmvTimer tm;
  if (timed) tm.begin(s);
  if (tv)
    e = gauss ? launch_kmvtc5_tv_gauss(nh, csep, M, variant, g.G, smem, s, R.ma5, P.mb5, args)
              : launch_kmvtc5_tv_matern(nh, csep, M, variant, g.G, smem, s, R.ma5, P.mb5, args);
  else
    e = gauss ? launch_kmvtc5_gauss(nh, csep, M, variant, g.G, smem, s, R.ma5, P.mb5, args)
              : launch_kmvtc5_matern(nh, csep, M, variant, g.G, smem, s, R.ma5, P.mb5, args);
  if (timed) tm.end(s);
  count_launch();
  return e;
}

// Variant for this product: forced, cached, tuned now, or the default.
template <typename TV5>
static int choose_variant(const PointsF32 &R, const PointsF32 &P, bool square, int M,
                          const TV5 *Vg,
                          int64_t ldv, int mg, DevBuf<float> &part, int *fault, cudaStream_t s,
                          bool quiet) {
  const int forced = g_t5_variant.load();
  if (forced > 0 && t5_variant_valid(forced, M, square)) return forced;
  if (quiet) return t5_default_variant(P, M, square);
  const auto key = std::make_tuple(P.kern, P.nh5, P.csep5, M, R.N, P.N, square);
  {
    std::lock_guard<std::mutex> lk(g_t5_mtx);
    auto it = g_t5_tuned.find(key);
    if (it != g_t5_tuned.end()) return it->second.best;
  }
  if (!autotune_on()) return t5_default_variant(P, M, square);
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(s, &cap) != cudaSuccess || cap != cudaStreamCaptureStatusNone)
    return t5_default_variant(P, M, square);   // timing would synchronise a capturing stream
  cudaEvent_t e0 = nullptr, e1 = nullptr;
  if (cudaEventCreate(&e0) != cudaSuccess || cudaEventCreate(&e1) != cudaSuccess) {
    if (e0) cudaEventDestroy(e0);
    cudaGetLastError();
    return t5_default_variant(P, M, square);
  }
  T5Tune tune;
  float best_ms = 1e30f;
  tune.best = t5_default_variant(P, M, square);
  for (int v = 1; v <= T5_NVARIANTS; ++v) {
    if (!t5_variant_valid(v, M, square)) continue;
    const T5Geometry g = t5_geometry(R.N, P.N, t5_variant_tn(v));
    const size_t need = t5_scratch_floats(g, M);
    if (part.n < need && part.alloc(need, s) != KRR_OK) break;
    float ms = 0.0f;
    bool ok = true;
    for (int rep = 0; rep < 2 && ok; ++rep) {   // the second launch is timed
      ok = t5_launch(R, P, M, v, g, Vg, ldv, mg, part.p, fault, nullptr, s, false) == cudaSuccess &&
           cudaEventRecord(e0, s) == cudaSuccess &&
           t5_launch(R, P, M, v, g, Vg, ldv, mg, part.p, fault, nullptr, s, false) == cudaSuccess &&
           cudaEventRecord(e1, s) == cudaSuccess && cudaEventSynchronize(e1) == cudaSuccess &&
           cudaEventElapsedTime(&ms, e0, e1) == cudaSuccess;
    }
    if (!ok) {
      cudaGetLastError();
      continue;
    }
    tune.ms[v] = ms;
    if (ms < best_ms) {
      best_ms = ms;
      tune.best = v;
    }
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  std::lock_guard<std::mutex> lk(g_t5_mtx);
  g_t5_tuned[key] = tune;
  return tune.best;
}

template <typename TV5>
static krr_status tc5_products(const PointsF32 &R, const PointsF32 &P, double lambda, bool square,
                               const TV5 *V, int64_t ldv, int m, TV5 *Y, int64_t ldy,
                               cudaStream_t s, DevBuf<float> &part, bool quiet, int *flags) {
  const int64_t Nr = R.N, Nc = P.N;
  if (Nr == 0 || Nc == 0 || m == 0) return KRR_OK;
  KRR_REQUIRE(R.nh5 > 0 && P.nh5 == R.nh5 && P.csep5 == R.csep5 && R.kern == P.kern,
              "tcgen05 product: operands missing or of different layouts");
  int *fault = tc5_fault_ptr();
  KRR_REQUIRE(fault != nullptr, "tcgen05 product: no fault flag on this device");
  // One launch of 16 where two of 8 would both take their sums on the tensor
  // cores: the kernel values, their split and the distances are formed once.
  // N = 50021, d = 32, Matern, m = 16: 2.93 -> 1.79 ms (N = 1e5, d = 16,
  // Gaussian: 5.9 -> 4.2 ms).  From 9 to 12 a launch of 8 and
  // one of 4 keep the float32 sums of the latter.
  const int forced = g_t5_variant.load();
  const bool wide = square && (forced == 0 || forced == 8 || forced == 9);
  int mg = 0;
  for (int c0 = 0; c0 < m; c0 += mg) {
    mg = std::min(wide && m - c0 > 12 ? 16 : 8, m - c0);
    const int M = mg <= 2 ? 2 : mg <= 4 ? 4 : mg <= 8 ? 8 : 16;
    const TV5 *Vg = V + (int64_t)c0 * ldv;
    const int variant = choose_variant(R, P, square, M, Vg, ldv, mg, part, fault, s, quiet);
    const T5Geometry g = t5_geometry(Nr, Nc, t5_variant_tn(variant));
    const size_t need = t5_scratch_floats(g, M);
    if (part.n < need) KRR_TRY(part.alloc(need, s));
    cudaError_t e = t5_launch(R, P, M, variant, g, Vg, ldv, mg, part.p, fault, flags, s, !quiet);
    if (e != cudaSuccess) {
      set_error("tcgen05 product launch failed: %s", cudaGetErrorString(e));
      return KRR_ECUDA;
    }
    const int CG = t5_variant_ew(variant) / 4;
    const int *vexp = t5_variant_tv(variant) ? t5_vexp(part.p, g, M) : nullptr;
    const TV5 *Vs = square ? Vg : nullptr;
    TV5 *Yg = Y + (int64_t)c0 * ldy;
    // more than four CTAs a row block: the grouped sum
    if ((int64_t)g.C * g.G > 4 * g.T)
      t5_reduce_many_kernel<TV5><<<dim3(ceil_div(Nr, 32), mg), 32 * T5_RED_WARPS, 0, s>>>(
          part.p, Nr, mg, M, g.C, g.T, g.G, g.J, CG, vexp, lambda, Vs, ldv, Yg, ldy, fault, flags);
    else
      t5_reduce_kernel<TV5><<<ceil_div(Nr, 256), 256, 0, s>>>(
          part.p, Nr, mg, M, g.C, g.T, g.G, g.J, CG, vexp, lambda, Vs, ldv, Yg, ldy, fault, flags);
    KRR_LAUNCH_CHECK();
  }
  return KRR_OK;
}

krr_status kmv_tc5(const PointsF32 &R, const PointsF32 &P, float lambda, bool square,
                   const float *V, int64_t ldv, int m, float *Y, int64_t ldy, cudaStream_t s,
                   DevBuf<float> &part, bool quiet) {
  return tc5_products<float>(R, P, (double)lambda, square, V, ldv, m, Y, ldy, s, part, quiet,
                             nullptr);
}

krr_status kmv_tc5_call(const double *Xr, int64_t Nr, const double *Xd, int64_t N, int d,
                        int kern, double sigma, double lambda, const double *V, int m, double *Y,
                        cudaStream_t s, bool *done) {
  *done = false;
  if (product_path() != 0 || kern == KLAPLACE || d > 32) return KRR_OK;
  PointsF32 P, R;
  auto set = [&](PointsF32 &Q, int64_t n) {
    Q.dp = (d + 3) / 4 * 4;
    Q.d = d;
    Q.N = n;
    Q.kern = kern;
    Q.sigma = sigma;
  };
  set(P, N);
  DevBuf<int> flags;
  KRR_TRY(flags.alloc(2, s));
  KRR_TRY(points_mean(Xd, N, d, s, P.mean, flags.p));
  KRR_TRY(tc5_operands(Xd, s, P, P.mean.p, Xr == nullptr, true, flags.p));
  if (Xr) {
    set(R, Nr);
    KRR_TRY(tc5_operands(Xr, s, R, P.mean.p, true, false, flags.p));
  }
  DevBuf<float> part;
  // the shift as the float32 products apply it
  KRR_TRY(tc5_products<double>(Xr ? R : P, P, (double)(float)lambda, Xr == nullptr, V, N, m, Y,
                               Xr ? Nr : N, s, part, false, flags.p));
  int h[2] = {0, 0};
  KRR_CUDA_TRY(cudaMemcpyAsync(h, flags.p, sizeof(h), cudaMemcpyDeviceToHost, s));
  KRR_CUDA_TRY(cudaStreamSynchronize(s));
  if (h[1]) return tc5_check_fault(s);
  *done = h[0] == 0;
  return KRR_OK;
}

}  // namespace krr
