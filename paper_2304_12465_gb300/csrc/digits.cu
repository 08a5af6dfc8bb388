// C -= A B^T by digits on the fifth-generation tensor cores (digits.cuh): the
// Schur update of Alg. 3 and the off-diagonal part of its triangular solve.
#include <algorithm>

#include "blackwell.cuh"
#include "dense.cuh"
#include "digits.cuh"
#include "kmv.cuh"

namespace krr {

constexpr int DG_ROWS = 128;       // rows of C per CTA (TMEM lanes)
constexpr int DG_WORKERS = 8;      // warps that convert A and read the sums out
constexpr int DG_THREADS = (DG_WORKERS + 2) * 32;
constexpr int DG_ADIG = DG_ROWS * 32;           // bytes of one digit of 128 x 16 of A
constexpr int DG_LOWSTEPS = DIG_LOW / 16;       // steps of 16 terms between read-outs
constexpr int DG_HIGHCHUNKS = DIG_HIGH / DIG_LOW;
constexpr long long DG_WAIT_BUDGET = 1LL << 32;   // about 2 s

// Columns of one group: 64, or what is left rounded up to 16.
__host__ __device__ constexpr int dg_group_cols(int nc, int g) {
  return nc - 64 * g >= 64 ? 64 : (nc - 64 * g + 15) / 16 * 16;
}
// Instances for up to NC columns: stages of the ring, TMEM columns.
__host__ __device__ constexpr int dg_stages(int NC) { return NC == 32 ? 2 : 4; }
__host__ __device__ constexpr int dg_stage_bytes(int NC) { return DIG_N * (DG_ADIG + NC * 32); }
// Steps of A in flight to shared memory, 16 KB each (a thread's own entries).
__host__ __device__ constexpr int dg_ahead(int NC) { return NC == 32 ? 2 : 3; }
constexpr int DG_AHEAD_BYTES = DG_WORKERS * 32 * 8 * 8;
constexpr size_t dg_smem(int NC) {
  return 1024 + (size_t)dg_stages(NC) * dg_stage_bytes(NC) +
         (size_t)dg_ahead(NC) * DG_AHEAD_BYTES + 8 * (3 * dg_stages(NC) + 3) + 16;
}

// Digits of B (nc rows of K entries: row c at B + rows[c] (rows NULL: c), step
// ldb between entries) as the kernel's shared tiles hold them: for column group
// g and step of 16 terms, the seven digits one after the other, each a
// K-major operand of dg_group_cols rows of 32 bytes in the 32-byte swizzle
// (zero padded).  A thread makes half a row.  n2: squared norms of the rows,
// indexed like them; their scales go to shift.
__global__ void dig_rows_kernel(const double *__restrict__ B, int64_t ldb,
                                const int64_t *__restrict__ rows,
                                const double *__restrict__ n2, int nc, int K, int K16,
                                uint4 *__restrict__ img, int *__restrict__ shift) {
  const int ncp = (nc + 15) / 16 * 16;
  const int64_t total = (int64_t)K16 * ncp * 2;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total;
       e += (int64_t)gridDim.x * blockDim.x) {
    const int c = (int)(e % ncp), half = (int)((e / ncp) & 1);
    const int step = (int)(e / ncp / 2);
    const int k = step * 16 + half * 8;
    double x[8];
    const int64_t r = c < nc ? (rows ? rows[c] : c) : 0;
    const int sh = c < nc ? dig_shift(n2[r]) : 0;
    if (step == 0 && half == 0) shift[c] = sh;
#pragma unroll
    for (int t = 0; t < 8; ++t)
      x[t] = (c < nc && k + t < K) ? B[r + (int64_t)(k + t) * ldb] : 0.0;
    uint32_t d[4][DIG_N];
#pragma unroll
    for (int t = 0; t < 4; ++t) dig_pair(x[2 * t], x[2 * t + 1], 1023 - sh, d[t]);
    const int g = c / 64, n = c % 64, ncol = dg_group_cols(nc, g);
    uint4 *dst = img + ((int64_t)g * K16 * 64 + (int64_t)step * ncol) * DIG_N * 2;
#pragma unroll
    for (int s = 0; s < DIG_N; ++s)
      dst[(s * ncol + n) * 2 + (half ^ ((n >> 2) & 1))] =
          make_uint4(d[0][s], d[1][s], d[2][s], d[3][s]);
  }
}

// C (N x nc, ldc) -= A (N x K, lda) B^T, B and its scales as dig_rows_kernel lays
// them out, an2 the squared norms of A's rows; cmap (optional) gives the column of
// C for each row of B.  A CTA takes 128 rows and
// one group of up to NC columns (blockIdx.x: groups of a row tile next to one
// another, so that the second one finds its rows of A in L2).
//
// Warps 0-7 convert A, read column by column (256-byte segments, copied two or
// three steps ahead to shared memory by the thread that will use them, since
// eight warps with the loads in registers waited for them): a thread makes the
// seven digits of eight entries of a row, 16 bytes each, into a ring of stages
// in the MMAs' K-major layout; a producer lane copies B's digits beside them.
// One lane issues the MMAs: digit s of A times digits 0 .. 6 - s of B, which lie
// one after the other as rows of one operand and whose products go to groups s
// .. 6, adjacent in TMEM: ten MMAs a step instead of 28, N up to 256.  Every DIG_LOW terms the eight warps add the
// accumulators to their 64-bit totals in registers (32 a thread); the ring's
// stages are filled before, so that the MMAs go on at once.
//
// A step of 64 columns takes about 900 clocks at the MMAs' rate (0.40 ms for N =
// 1e5, K = 900, 100 columns with the conversion taken out) and as many issue
// slots a scheduler to convert, with eight warps to fill them (0.8 ms with the
// MMAs taken out).  Measured at N = 1e5, 100 columns: 0.51 ms for K = 500 and
// 0.83 ms for K = 900, against 1.04 and 1.75 ms for the same digits with
// mma.sync, and 3.35 and 5.87 ms for a float-float product on the float32 pipe;
// with A's entries loaded to registers two steps ahead 0.54 and 0.88 ms, and C
// read and written entry by entry 0.1 ms more.  Up to 32 columns two CTAs share
// an SM (45 us at N = 1e5, K = 20 to 80, where mma.sync took 57).
template <int NC>
__global__ void __launch_bounds__(DG_THREADS, NC == 32 ? 2 : 1)
dig_gemm_kernel(const double *__restrict__ A, int64_t lda, int64_t N, int K,
                const double *__restrict__ an2, const uint4 *__restrict__ img,
                const int *__restrict__ bshift, int nc, int groups, double *__restrict__ C,
                int64_t ldc, const int *__restrict__ cmap, int *fault) {
  constexpr int ST = dg_stages(NC);
  constexpr int STAGE = dg_stage_bytes(NC);
  constexpr int AHEAD = dg_ahead(NC);
  constexpr int TCOLS = NC == 32 ? 256 : 512;
  constexpr int BAR_A = 0, BAR_B = ST, BAR_E = 2 * ST, BAR_D = 3 * ST, BAR_R = 3 * ST + 1,
                BAR_FIN = 3 * ST + 2;
  extern __shared__ uint8_t dg_raw[];
  const uint32_t raw = bw::smem_u32(dg_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;
  const uint32_t sX = base + ST * STAGE;   // [AHEAD][8 entries][256 threads] of A
  const uint32_t sBar = sX + AHEAD * DG_AHEAD_BYTES;
  uint32_t *tslot = reinterpret_cast<uint32_t *>(dg_raw + (sBar - raw) + 8 * (3 * ST + 3));
  volatile int *abort_flag = reinterpret_cast<volatile int *>(tslot + 1);
  auto bar = [&](int i) -> uint32_t { return sBar + 8u * (uint32_t)i; };

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int grp = (int)(blockIdx.x % groups);
  const int64_t row0 = (int64_t)(blockIdx.x / groups) * DG_ROWS;
  const int ncol = dg_group_cols(nc, grp);
  const int K16 = (K + 15) / 16;
  const int chunks = (K16 + DG_LOWSTEPS - 1) / DG_LOWSTEPS;

  if (threadIdx.x == 0) {
    for (int s = 0; s < ST; ++s) {
      bw::mbar_init(bar(BAR_A + s), DG_WORKERS);
      bw::mbar_init(bar(BAR_B + s), 1);
      bw::mbar_init(bar(BAR_E + s), 1);
    }
    bw::mbar_init(bar(BAR_D), 1);
    bw::mbar_init(bar(BAR_R), DG_WORKERS);
    bw::mbar_init(bar(BAR_FIN), 1);
    *abort_flag = 0;
    bw::fence_mbar_init();
  }
  if (warp == DG_WORKERS + 1) {
    bw::tmem_alloc(bw::smem_u32(tslot), TCOLS);
    bw::tmem_relinquish();
  }
  bw::tc_fence_before();
  __syncthreads();
  bw::tc_fence_after();
  const uint32_t tmem = *tslot;
  // bounded wait; on timeout records the fault and aborts the CTA
  auto wait = [&](int i, uint32_t parity) -> bool {
    if (bw::mbar_wait_abortable(bar(i), parity, DG_WAIT_BUDGET, abort_flag)) return true;
    *abort_flag = 1;
    atomicOr(fault, 1);
    return false;
  };

  if (warp == DG_WORKERS) {
    // ---------------------------------------------------------- B's digits
    if (lane == 0) {
      const uint32_t bytes = (uint32_t)(DIG_N * ncol * 32);
      const uint4 *src = img + (int64_t)grp * K16 * 64 * DIG_N * 2;
      int issued = 0, s = 0;
      uint32_t ph = 0;
      for (int step = 0; step < K16; ++step) {
        if (!wait(BAR_E + s, ph ^ 1u)) break;
        bw::mbar_arrive_expect_tx(bar(BAR_B + s), bytes);
        bw::bulk_load(base + (uint32_t)(s * STAGE + DIG_N * DG_ADIG),
                      src + (int64_t)step * ncol * DIG_N * 2, bytes, bar(BAR_B + s));
        ++issued;
        if (++s == ST) s = 0, ph ^= 1u;
      }
      // wait (bounded, quietly) for the copies in flight
      for (int q = issued > ST ? issued - ST : 0; q < issued; ++q)
        bw::mbar_wait(bar(BAR_B + q % ST), (uint32_t)((q / ST) & 1), DG_WAIT_BUDGET >> 4);
    }
    __syncwarp();
  } else if (warp == DG_WORKERS + 1) {
    // ----------------------------------------------------------------- MMA
    if (lane == 0) {
      int s = 0, in = 0, chunk = 0;
      uint32_t ph = 0;
      for (int step = 0; step < K16; ++step) {
        // the sums of the chunk before have been read out
        if (in == 0 && chunk > 0 && !wait(BAR_R, (uint32_t)((chunk - 1) & 1))) break;
        if (!wait(BAR_A + s, ph) || !wait(BAR_B + s, ph)) break;
        bw::tc_fence_after();
        const uint32_t a0 = base + (uint32_t)(s * STAGE), b0 = a0 + DIG_N * DG_ADIG;
        auto mma = [&](int sa, int t, int nt, uint32_t acc) {
          bw::mma_f16(tmem + (uint32_t)((sa + t) * ncol),
                      bw::sdesc_kmajor_sw32(a0 + sa * DG_ADIG),
                      bw::sdesc_kmajor_sw32(b0 + (uint32_t)(t * ncol * 32)),
                      bw::idesc_f16_f32(DG_ROWS, nt * ncol), acc);
        };
        // groups 0..2 and 3..6 start anew after their read-outs
        mma(0, 0, 3, (in == 0 && chunk % DG_HIGHCHUNKS == 0) ? 0u : 1u);
        mma(0, 3, 4, in == 0 ? 0u : 1u);
        mma(1, 0, 3, 1);
        mma(1, 3, 3, 1);
        mma(2, 0, 3, 1);
        mma(2, 3, 2, 1);
        mma(3, 0, 4, 1);
        mma(4, 0, 3, 1);
        mma(5, 0, 2, 1);
        mma(6, 0, 1, 1);
        bw::mma_commit(bar(BAR_E + s));
        if (++in == DG_LOWSTEPS || step + 1 == K16) {
          bw::mma_commit(bar(BAR_D));
          in = 0;
          ++chunk;
        }
        if (++s == ST) s = 0, ph ^= 1u;
      }
      // every MMA issued so far has completed once FIN flips
      bw::mma_commit(bar(BAR_FIN));
      bw::mbar_wait(bar(BAR_FIN), 0, DG_WAIT_BUDGET >> 4);
    }
    __syncwarp();
  } else {
    // ------------------------------------------- conversion and read-outs
    const int half = warp >> 2;               // entries 8 half .. + 7, columns of half
    const int rl = (warp & 3) * 32 + lane;    // row of the tile, TMEM lane
    const int64_t row = row0 + rl;
    const bool ok = row < N;
    const int top = 1023 - (ok ? dig_shift(an2[row]) : 0);
    const int nc2 = ncol / 2;
    const double *Ar = A + row + (int64_t)(8 * half) * lda;
    const uint32_t dst = base + (uint32_t)(rl * 32 + ((half ^ ((rl >> 2) & 1)) * 16));
    const uint32_t xs = sX + (uint32_t)threadIdx.x * 8;
    auto load = [&](int step, int slot) {
      if (step < K16) {
#pragma unroll
        for (int t = 0; t < 8; ++t) {
          const bool in = ok && step * 16 + 8 * half + t < K;
          asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(
                           xs + (uint32_t)(slot * DG_AHEAD_BYTES + t * DG_WORKERS * 32 * 8)),
                       "l"(in ? Ar + (int64_t)(step * 16 + t) * lda : A), "r"(in ? 8 : 0)
                       : "memory");
        }
      }
      asm volatile("cp.async.commit_group;" ::: "memory");
    };
    int64_t tot[NC / 2];
#pragma unroll
    for (int i = 0; i < NC / 2; ++i) tot[i] = 0;
    const uint32_t tcol = tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)(half * nc2);
    auto read_out = [&](int chunk) -> bool {
      if (!__all_sync(0xffffffffu, wait(BAR_D, (uint32_t)(chunk & 1)))) return false;
      bw::tc_fence_after();
      const bool high = (chunk + 1) % DG_HIGHCHUNKS == 0 || chunk + 1 == chunks;
#pragma unroll
      for (int cb = 0; cb < NC / 16; ++cb) {
        if (cb * 8 < nc2) {
          uint32_t r[32];
#pragma unroll
          for (int g = 3; g < 7; ++g)
            bw::tmem_ld_32x32b_x8(tcol + (uint32_t)(g * ncol + cb * 8), r + (g - 3) * 8);
          bw::tmem_wait_ld32(r);
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            // units 2^-64, exact
            const int64_t lo = ((int64_t)__float2int_rn(__uint_as_float(r[i])) << 24) +
                               ((int64_t)__float2int_rn(__uint_as_float(r[8 + i])) << 16) +
                               ((int64_t)__float2int_rn(__uint_as_float(r[16 + i])) << 8) +
                               (int64_t)__float2int_rn(__uint_as_float(r[24 + i]));
            tot[cb * 8 + i] += (lo + 8) >> 4;
          }
          if (high) {
#pragma unroll
            for (int g = 0; g < 3; ++g)
              bw::tmem_ld_32x32b_x8(tcol + (uint32_t)(g * ncol + cb * 8), r + g * 8);
            bw::tmem_wait_ld32(r);
#pragma unroll
            for (int i = 0; i < 8; ++i) {
              // units 2^-32
              const int64_t hi = ((int64_t)__float2int_rn(__uint_as_float(r[i])) << 16) +
                                 ((int64_t)__float2int_rn(__uint_as_float(r[8 + i])) << 8) +
                                 (int64_t)__float2int_rn(__uint_as_float(r[16 + i]));
              tot[cb * 8 + i] += hi * (1ll << 28);
            }
          }
        }
      }
      bw::tc_fence_before();
      __syncwarp();
      if (lane == 0) bw::mbar_arrive(bar(BAR_R));
      return true;
    };
    int s = 0, chunk = 0, slot = 0;
    uint32_t ph = 0;
    bool good = true;
#pragma unroll
    for (int q = 0; q < AHEAD; ++q) load(q, q);
    for (int step = 0; step < K16; ++step) {
      // the ring is full of the next chunk's steps: the chunk before is read
      // out now, since the MMAs that would free a stage wait for it
      if (step == (chunk + 1) * DG_LOWSTEPS + ST) good = good && read_out(chunk++);
      good = good && __all_sync(0xffffffffu, wait(BAR_E + s, ph ^ 1u));
      if (!good) break;
      asm volatile("cp.async.wait_group %0;" ::"n"(AHEAD - 1) : "memory");
      double x[8];
#pragma unroll
      for (int t = 0; t < 8; ++t)
        asm volatile("ld.shared.f64 %0, [%1];"
                     : "=d"(x[t])
                     : "r"(xs + (uint32_t)(slot * DG_AHEAD_BYTES + t * DG_WORKERS * 32 * 8))
                     : "memory");
      load(step + AHEAD, slot);
      uint32_t d[4][DIG_N];
#pragma unroll
      for (int t = 0; t < 4; ++t) dig_pair(x[2 * t], x[2 * t + 1], top, d[t]);
#pragma unroll
      for (int q = 0; q < DIG_N; ++q)
        asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(
                         dst + (uint32_t)(s * STAGE + q * DG_ADIG)),
                     "r"(d[0][q]), "r"(d[1][q]), "r"(d[2][q]), "r"(d[3][q])
                     : "memory");
      bw::fence_async_shared();
      __syncwarp();
      if (lane == 0) bw::mbar_arrive(bar(BAR_A + s));
      if (++s == ST) s = 0, ph ^= 1u;
      if (++slot == AHEAD) slot = 0;
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
    while (good && chunk < chunks) good = read_out(chunk++);
    if (good && ok) {
      // eight columns of C at a time, all read before the first is written
#pragma unroll
      for (int cb = 0; cb < NC / 16; ++cb) {
        const int c0 = grp * 64 + half * nc2 + cb * 8;
        if (cb * 8 < nc2) {
          double *p[8], v[8];
          int sb[8];
#pragma unroll
          for (int i = 0; i < 8; ++i)
            if (c0 + i < nc) {
              p[i] = C + row + (int64_t)(cmap ? cmap[c0 + i] : c0 + i) * ldc;
              v[i] = *p[i];
              sb[i] = bshift[c0 + i];
            }
#pragma unroll
          for (int i = 0; i < 8; ++i)
            if (c0 + i < nc)   // the total's unit is 2^(-60 - the two rows' scales)
              *p[i] = v[i] - (double)tot[cb * 8 + i] *
                                 __hiloint2double((top - 60 - sb[i]) << 20, 0);
        }
      }
    }
  }
  bw::tc_fence_before();
  __syncthreads();
  if (warp == DG_WORKERS + 1) {
    bw::tc_fence_after();
    bw::tmem_dealloc(tmem, TCOLS);
  }
}

// B's digits, then its scales.
size_t dig_image_bytes(int nc, int K) {
  return (size_t)((K + 15) / 16 * DIG_N * 32 + 4) * ((nc + 15) / 16 * 16);
}

template <int NC>
static krr_status launch_dig(const double *A, int64_t lda, int64_t N, int K, const double *an2,
                             const uint4 *img, const int *bshift, int nc, double *C, int64_t ldc,
                             const int *cmap, int *fault, cudaStream_t s) {
  KRR_TRY(raise_smem_limit(dig_gemm_kernel<NC>, dg_smem(NC)));
  const int groups = (nc + 63) / 64;
  dig_gemm_kernel<NC><<<(unsigned)(ceil_div(N, DG_ROWS) * groups), DG_THREADS, dg_smem(NC), s>>>(
      A, lda, N, K, an2, img, bshift, nc, groups, C, ldc, cmap, fault);
  KRR_LAUNCH_CHECK();
  return KRR_OK;
}

krr_status dig_gemm_sub(const double *A, int64_t lda, int64_t N, int K, const double *an2,
                        const double *B, int64_t ldb, const int64_t *rows, const double *bn2,
                        int nc, double *C, int64_t ldc, const int *cmap, uint4 *img,
                        cudaStream_t s) {
  if (N <= 0 || K <= 0 || nc <= 0) return KRR_OK;
  int *fault = tc5_fault_ptr();
  KRR_REQUIRE(fault != nullptr, "digit product: no fault flag on this device");
  const int K16 = (K + 15) / 16, ncp = (nc + 15) / 16 * 16;
  int *bshift = reinterpret_cast<int *>(img + (size_t)K16 * DIG_N * 2 * ncp);
  const int64_t total = (int64_t)K16 * ncp * 2;
  dig_rows_kernel<<<(unsigned)std::min<int64_t>((total + 127) / 128, 4 * num_sms()), 128, 0, s>>>(
      B, ldb, rows, bn2, nc, K, K16, img, bshift);
  KRR_LAUNCH_CHECK();
  if (nc <= 32)
    return launch_dig<32>(A, lda, N, K, an2, img, bshift, nc, C, ldc, cmap, fault, s);
  return launch_dig<64>(A, lda, N, K, an2, img, bshift, nc, C, ldc, cmap, fault, s);
}

}  // namespace krr
