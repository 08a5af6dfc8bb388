// Fused product Y = K(rows, columns) V (+ lambda V for the square product)
// for the Gaussian and Matern kernels (Sec. 2.1; the "Product" primitive of
// Alg. 1), with the inner products x_i . x_j on the fifth-generation tensor
// cores (tcgen05.mma, accumulators in Tensor Memory) and the kernel values
// and sums over V in float32 registers.
//
// Arithmetic.  Points are centred and scaled as for the float32 FMA product,
// so that kappa = 2^D (Gaussian) or D = -q^2/2 (Matern) with
// D = x_i . x_j + c_i + c_j and c = -|x|^2 / 2; the Gaussian's operands carry
// c + 7 instead of c, so that its D is log2 kappa + 14 and ex2 gives the
// kernel value scaled by 2^14 (the FMA variants multiply by V scaled by
// 2^-14, exactly; the TV variants need the headroom).  Each coordinate is split
// into two halves x = h + l (h = fp16(x), l = fp16(x - h), |x - h - l| <=
// 2^-22 |x|) and c into three fp16 pieces c1 + c2 + c3.  Each point has
// 16-wide K-blocks [H_0..H_{NH-1} | L_0..L_{NH-1} | C], stored K-block-major
// (kb x N x 16 halves) so that one column tile is a single 3-D TMA box of
// contiguous 4 KB slabs:
// the row operand's c-part is (c1, c2, c3, 1, 1, 1) and the column operand's
// (1, 1, 1, c1, c2, c3), so the product of the two c-parts is c_i + c_j.  The
// c-part sits in a block of its own (CSEP = 1) or in the unused positions
// 10..15 of the last H block (CSEP = 0, when d mod 16 is 1..10).  D is then
// the float32 sum of the MMAs (L_i, H_j), (H_i, L_j), (C_i, C_j), (H_i, H_j)
// over the coordinate blocks, small terms first; the dropped l_i . l_j is
// below 2^-22 |x_i| |x_j|.
//
// Decomposition.  A row block is 256 rows (two row tiles of 128 = the TMEM
// lanes), a column tile 128 columns (the MMA's N).  The (row block, column
// tile) pairs are numbered row-block-major and CTA b of G persistent CTAs
// (one per SM) takes the contiguous range [b T / G, (b + 1) T / G), so the
// load is balanced to one tile.  Its pairs fall into segments, one per row
// block it touches; each segment's partial sums go to part[b][j] (j the
// segment's index within the CTA) and t5_reduce_kernel adds, for every row,
// the segments of the CTAs that cover its row block in CTA order (a fixed
// order: results are deterministic for a given grid).
//
// Warp roles (320 threads):
//   warp 8 (producer): one lane issues the TMA loads of the row operand (both
//     row tiles, once per segment) and of each column tile's operand into a
//     ring of t5_stages(kb, M) stages (up to 8), plus a bulk copy of the tile's
//     right-hand sides, prepared once per product (t5_vpair_kernel,
//     t5_vfrag_kernel), all completing on the stage's barrier.
//   warp 9 (MMA): allocates all 512 TMEM columns; one lane issues, per column
//     tile and row tile, the MMAs of D into one of two accumulator buffers
//     (2 buffers x 2 row tiles x 128 columns), and commits them to the
//     barriers that release the column stage and hand the buffer to the
//     epilogue.
//   warps 0-7 (epilogue; 12 or 16 in other variants): warps 0-3 take the even
//     tiles and warps 4-7 the odd ones.  Warp w reads TMEM lanes 32 (w % 4) ..
//     + 31 with tcgen05.ld 32x32b, 16 columns of both row tiles at a time: a
//     lane holds one row of each row tile, forms kappa with ex2 on the MUFU and
//     accumulates V with FFMA2 over pairs of columns of one row, so that V is
//     read undoubled, as warp-wide broadcasts, and sums need no shuffles.
//
// What bounds it (N = 1e5, d = 16, m = 4, 1e10 entries, 2.15 ms): FFMA2, ex2
// and the issue slots each need 1.0-1.1 ms; the hand-over of a tile costs an
// epilogue warp about 700 cycles, measured with the work itself taken out, and
// the eight MMAs 510.  With all eight warps on every tile these were waits of
// both warps of a scheduler at once; alternate tiles let one warp compute
// meanwhile.  Against a layout of eight rows a lane (16x256b), V doubled and
// every warp on every tile: m = 4 2.30 -> 2.15 ms, m = 2 1.75 -> 1.61 (16
// warps), m = 8 without tensor-core sums 4.35 -> 3.59, Matern m = 4 4.74 ->
// 4.35 (16 warps).  Taken with alternate tiles too, eight rows a lane
// and column pairs need a quarter of the V loads but 168 registers: 2.27 ms.
//
// Every mbarrier wait is bounded (T5_WAIT_BUDGET cycles); a wait that gives
// up sets *fault, raises a CTA-wide abort flag so the other roles leave too,
// and the CTA waits (bounded) for its own TMA copies and MMAs in flight and
// frees its Tensor Memory before returning.
#pragma once

#include <cuda_fp16.h>

#include "blackwell.cuh"
#include "kmv_kernels.cuh"

namespace krr {

constexpr int T5_TM = 128;                   // rows of a row tile (TMEM lanes)
constexpr int T5_RT = 2;                     // row tiles per row block
constexpr int T5_RB = T5_TM * T5_RT;         // rows per row block
constexpr int T5_TN = 128;                   // columns per column tile (MMA N)
constexpr int T5_BLK = T5_TM * 32;           // bytes of one 16-wide K-block of 128 points
constexpr int T5_TMEM_COLS = 512;
constexpr long long T5_WAIT_BUDGET = 1LL << 32;   // about 2 s at 2 GHz
constexpr float T5_MAX_COORD = 16384.0f;     // |scaled coordinate| bound of the split
constexpr float T5_MAX_C = 32768.0f;         // |c| bound of its fp16 pieces

// K-blocks of the split layout for dimension d.
__host__ __device__ constexpr int t5_nh(int d) { return (d + 15) / 16; }
__host__ __device__ constexpr int t5_csep(int d) { return (d % 16 == 0 || d % 16 > 10) ? 1 : 0; }
__host__ __device__ constexpr int t5_kb(int nh, int csep) { return 2 * nh + csep; }

// B fragments of 8 slots per batch of 16 columns (TV variants).
__host__ __device__ constexpr int t5_nfrag(int M) { return M >= 8 ? M / 4 : 1; }

// Floats of shared memory that hold the running totals of the TV variants at
// M = 16 (four fragments' accumulators of four row groups; totals in registers
// spilled 390 bytes).  0 otherwise: totals in registers.
__host__ __device__ constexpr int t5_tot_floats(int EW, int M, int TV) {
  return (TV && M == 16) ? EW * 32 * 16 * t5_nfrag(M) : 0;
}

// 16-byte words of right-hand sides per pair of columns: M / 2 of {v_c(j),
// v_c(j + 1), v_c+1(j), v_c+1(j + 1)} (FMA sums), or the B fragments (TV).
__host__ __device__ constexpr int t5_vwords(int M, int TV) { return TV ? 2 * t5_nfrag(M) : M / 2; }

// Shared-memory bytes of a stage's right-hand sides (enough for either).
__host__ __device__ constexpr int t5_vstage(int M) {
  return (t5_vwords(M, 1) > t5_vwords(M, 0) ? t5_vwords(M, 1) : t5_vwords(M, 0)) * T5_TN / 2 * 16;
}

// Column-tile pipeline stages: as many as fit (at most 8) in about 200 KB of
// shared memory beside the row operand and the totals, so that TMA latency is
// hidden.
__host__ __device__ constexpr int t5_stages(int kb, int M, int tot_floats = 0) {
  return ((204800 - 1024 - T5_RT * kb * T5_BLK - 4 * tot_floats) / (kb * T5_BLK + t5_vstage(M))) >
                 8
             ? 8
             : ((204800 - 1024 - T5_RT * kb * T5_BLK - 4 * tot_floats) /
                (kb * T5_BLK + t5_vstage(M)));
}

// Barrier indices in shared memory for ST stages.
__host__ __device__ constexpr int t5_bar_a_full() { return 0; }
__host__ __device__ constexpr int t5_bar_a_empty() { return 1; }
__host__ __device__ constexpr int t5_bar_b_full(int) { return 2; }
__host__ __device__ constexpr int t5_bar_b_empty(int st) { return 2 + st; }
__host__ __device__ constexpr int t5_bar_v_empty(int st) { return 2 + 2 * st; }
__host__ __device__ constexpr int t5_bar_d_full(int st) { return 2 + 3 * st; }
__host__ __device__ constexpr int t5_bar_d_empty(int st) { return 4 + 3 * st; }
__host__ __device__ constexpr int t5_bar_fin(int st) { return 6 + 3 * st; }
__host__ __device__ constexpr int t5_nbar(int st) { return 7 + 3 * st; }

// Shared memory of one CTA (bytes, including 1024 bytes of alignment slack).
__host__ __device__ constexpr int t5_smem_bytes(int kb, int M, int tot_floats = 0) {
  return 1024 + T5_RT * kb * T5_BLK +
         t5_stages(kb, M, tot_floats) * (kb * T5_BLK + t5_vstage(M)) + 4 * tot_floats +
         8 * t5_nbar(t5_stages(kb, M, tot_floats)) + 16;
}

struct T5Args {
  const float4 *v;      // right-hand sides of the column tiles (t5_vpair_kernel, t5_vfrag_kernel)
  int64_t Nc;           // column points
  float *part;          // G x J x (EW / 4) x M x T5_RB partial sums
  int C;            // column tiles
  int64_t T;        // row blocks x column tiles
  int J;            // segments per CTA (maximum)
  int *fault;       // set to 1 when a bounded wait gives up
  // optional: not zero when the points turned out not to fit the split (known
  // on the device before the host knows): every CTA then has no pairs
  const int *skip;
};

// Kernel values of the MMA accumulator D.
template <int KERN>
__device__ __forceinline__ float t5_kappa(uint32_t d) {
  return kappa_f32<KERN>(__uint_as_float(d));
}

// 2^14 kappa for the tensor-core sums (TV variants): the Gaussian's operands
// carry the factor in their c-parts (D = log2 kappa + 14), the Matern
// polynomial is scaled instead.
template <int KERN>
__device__ __forceinline__ float t5_kappa_scaled(uint32_t d) {
  if constexpr (KERN == KMATERN) {
    const float q = sqrt_approx(fmaxf(-2.0f * __uint_as_float(d), 0.0f));
    const float e = ex2_approx(-1.4426950408889634f * q);
    return fmaf(q, fmaf(q, 5461.3335f, 16384.0f), 16384.0f) * e;
  } else {
    return ex2_approx(__uint_as_float(d));
  }
}

// Splits two non-negative values k0, k1 into fp16 halves k = hi + lo: hi keeps
// the leading 11 significant bits (exact in fp16 for k >= 2^-14), lo = k - hi
// (exact in float32) rounded to fp16; packed with k0 in the low half.
__device__ __forceinline__ void t5_split_pair(float k0, float k1, uint32_t &hi, uint32_t &lo) {
  const float h0 = __uint_as_float(__float_as_uint(k0) & 0xFFFFE000u);
  const float h1 = __uint_as_float(__float_as_uint(k1) & 0xFFFFE000u);
  const float2 l = __ffma2_rn(f2(h0, h1), f2(-1.0f, -1.0f), f2(k0, k1));
  const __half2 hh = __floats2half2_rn(h0, h1), ll = __floats2half2_rn(l.x, l.y);
  hi = *reinterpret_cast<const uint32_t *>(&hh);
  lo = *reinterpret_cast<const uint32_t *>(&ll);
}

__device__ __forceinline__ void t5_mma_16816(float (&d)[4], const uint32_t (&a)[4], uint2 b) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, "
      "{%8,%9}, {%0,%1,%2,%3};\n"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b.x), "r"(b.y));
}

// Epilogue variants: EW epilogue warps (8, 12 or 16; TN the column tile: 128,
// or 96 for 12 warps, which share every tile), PIPE = 1 keeps the TMEM loads of the
// next 16 columns in flight while the current ones are computed, LAG = 1
// (with PIPE) software-pipelines the epilogue by one batch of 16 columns:
// the kernel values (ex2 on the MUFU) of batch b are formed while the FFMA2
// accumulation of batch b - 1 runs on the FMA pipe, across tile boundaries,
// so that the two pipes work at the same time instead of in turn.  TV = 1
// takes the sums over the right-hand sides on the tensor cores instead of the
// FMA pipe: the 16x256b TMEM layout of a batch of 16 columns is the A-operand
// fragment layout of mma.sync m16n8k16, so each kernel value, scaled by 2^14
// and split into fp16 halves hi + lo, enters two MMAs (A = hi, A = lo) whose
// B operand holds the right-hand sides split likewise, v s_c = v_hi + v_lo
// with a power-of-two scale s_c per right-hand side (t5_vfrag_kernel): B
// slots 0..M-1 the v_hi, M..2M-1 the v_lo (M <= 4), or one fragment of each
// for every eight right-hand sides (M = 8, 16).  Products of fp16 halves are exact in float32, so the result is
// (hi + lo)(v_hi + v_lo) summed in float32 per tile, then added to the
// segment total (two levels, as the FMA variants).
template <int KERN, int NH, int CSEP, int M, int EW, int PIPE, int LAG, int TN, int TV = 0>
__global__ void __launch_bounds__((EW + 2) * 32, 1)
kmvtc5_kernel(const __grid_constant__ CUtensorMap rowmap,
              const __grid_constant__ CUtensorMap colmap, const T5Args a) {
  // column tile of this variant (the MMA's N; the TMA box stays 128 points,
  // of which the first TN are used)
  constexpr int T5_TN = TN;
  constexpr int KB = 2 * NH + CSEP;
  constexpr int MP = M / 2;   // right-hand-side pairs
  constexpr int NB = t5_nfrag(M);        // B fragments per batch (TV)
  constexpr int VF = t5_vwords(M, TV) * T5_TN / 2;   // 16-byte right-hand-side words of a tile
  constexpr int TOTF = t5_tot_floats(EW, M, TV);     // running totals in shared memory
  constexpr int T5_ST = t5_stages(KB, M, TOTF);
  constexpr int T5_BAR_A_FULL = t5_bar_a_full();
  constexpr int T5_BAR_A_EMPTY = t5_bar_a_empty();
  constexpr int T5_BAR_B_FULL = t5_bar_b_full(T5_ST);
  constexpr int T5_BAR_B_EMPTY = t5_bar_b_empty(T5_ST);
  constexpr int T5_BAR_V_EMPTY = t5_bar_v_empty(T5_ST);
  constexpr int T5_BAR_D_FULL = t5_bar_d_full(T5_ST);
  constexpr int T5_BAR_D_EMPTY = t5_bar_d_empty(T5_ST);
  constexpr int T5_BAR_FIN = t5_bar_fin(T5_ST);
  constexpr int T5_NBAR = t5_nbar(T5_ST);
  constexpr int T5_EPI_WARPS = EW;
  // The two halves of 8 or 16 epilogue warps take alternate tiles (one D buffer
  // each), so that one half computes while the other hands over.
  // Not for the Matern tensor-core sums, whose warps issue without a pause (N =
  // 50021, d = 32, m = 8: 1.49 ms together, 1.56 in turn).
  constexpr int TG = EW % 8 == 0 && !(TV && KERN == KMATERN) ? 2 : 1;
  constexpr int T5_CG = EW / 4 / TG;            // column groups of a tile
  constexpr int T5_WCOLS = T5_TN / T5_CG;       // columns per epilogue warp per tile
  constexpr int T5_PRODUCER_WARP = EW;
  constexpr int T5_MMA_WARP = EW + 1;
  extern __shared__ uint8_t t5_smem[];
  const uint32_t raw = bw::smem_u32(t5_smem);
  const uint32_t base = (raw + 1023u) & ~1023u;
  uint8_t *gbase = t5_smem + (base - raw);
  const uint32_t sA = base;                                   // [rt][kb][128 x 32 B]
  const uint32_t sB = sA + T5_RT * KB * T5_BLK;               // [stage][kb][128 x 32 B]
  const uint32_t vOff = sB + T5_ST * KB * T5_BLK - base;
  float4 *sV = reinterpret_cast<float4 *>(gbase + vOff);       // [stage][VF]
  const uint32_t totOff = vOff + T5_ST * t5_vstage(M);
  float4 *sTot = reinterpret_cast<float4 *>(gbase + totOff);   // [warp][4 NB][32 lanes]
  const uint32_t sBar = base + totOff + 4 * TOTF;
  uint32_t *tslot = reinterpret_cast<uint32_t *>(gbase + (sBar - base) + 8 * T5_NBAR);
  volatile int *abort_flag = reinterpret_cast<volatile int *>(tslot + 1);
  auto bar = [&](int i) -> uint32_t { return sBar + 8u * (uint32_t)i; };

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int G = gridDim.x, b = blockIdx.x;
  const int64_t p_begin = (int64_t)b * a.T / G;
  const int64_t p_end = (a.skip && *a.skip) ? p_begin : (int64_t)(b + 1) * a.T / G;
  const int64_t rb_first = p_begin / a.C;
  const int ct_first = (int)(p_begin - rb_first * a.C);
  // (row block, column tile) of pair p are kept incrementally along the range
  // (no per-tile 64-bit division)

  if (threadIdx.x == 0) {
    bw::mbar_init(bar(T5_BAR_A_FULL), 1);
    bw::mbar_init(bar(T5_BAR_A_EMPTY), 1);
    for (int s = 0; s < T5_ST; ++s) {
      bw::mbar_init(bar(T5_BAR_B_FULL + s), 1);
      bw::mbar_init(bar(T5_BAR_B_EMPTY + s), 1);
      bw::mbar_init(bar(T5_BAR_V_EMPTY + s), T5_EPI_WARPS / TG);   // one arrival per warp
    }
    for (int i = 0; i < 2; ++i) {
      bw::mbar_init(bar(T5_BAR_D_FULL + i), 1);
      bw::mbar_init(bar(T5_BAR_D_EMPTY + i), T5_EPI_WARPS / TG);
    }
    bw::mbar_init(bar(T5_BAR_FIN), 1);
    *abort_flag = 0;
    bw::fence_mbar_init();
  }
  if (warp == T5_MMA_WARP) {
    bw::tmem_alloc(bw::smem_u32(tslot), T5_TMEM_COLS);
    bw::tmem_relinquish();
  }
  if (warp == T5_PRODUCER_WARP && lane == 0) {
    bw::prefetch_tensormap(&rowmap);
    bw::prefetch_tensormap(&colmap);
  }
  bw::tc_fence_before();
  __syncthreads();
  bw::tc_fence_after();
  const uint32_t tmem = *tslot;

  // bounded wait; on timeout records the fault and aborts the CTA
  auto wait = [&](int i, uint32_t parity) -> bool {
    if (bw::mbar_wait_abortable(bar(i), parity, T5_WAIT_BUDGET, abort_flag)) return true;
    *abort_flag = 1;
    atomicOr(a.fault, 1);
    return false;
  };

  if (warp == T5_PRODUCER_WARP) {
    // ------------------------------------------------------------ producer
    if (lane == 0) {
      constexpr uint32_t VBYTES = VF * 16;
      int64_t kt = 0, issued_b = 0;
      int issued_a = 0;
      int64_t rb = rb_first;
      int ct = ct_first;
      for (int64_t p = p_begin; p < p_end; ++p, ++kt, (++ct == a.C ? (ct = 0, ++rb) : 0)) {
        if (p == p_begin || ct == 0) {
          if (!wait(T5_BAR_A_EMPTY, (uint32_t)(issued_a & 1) ^ 1u)) break;
          bw::mbar_arrive_expect_tx(bar(T5_BAR_A_FULL), T5_RT * KB * T5_BLK);
#pragma unroll
          for (int rt = 0; rt < T5_RT; ++rt)
            bw::tma_load_3d(sA + rt * KB * T5_BLK, &rowmap, bar(T5_BAR_A_FULL), 0,
                            (int)(rb * T5_RB + rt * T5_TM), 0);
          ++issued_a;
        }
        const int s = (int)(kt % T5_ST);
        const uint32_t ph = (uint32_t)((kt / T5_ST) & 1);
        if (!wait(T5_BAR_B_EMPTY + s, ph ^ 1u) || !wait(T5_BAR_V_EMPTY + s, ph ^ 1u)) break;
        bw::mbar_arrive_expect_tx(bar(T5_BAR_B_FULL + s), KB * T5_BLK + VBYTES);
        bw::tma_load_3d(sB + s * KB * T5_BLK, &colmap, bar(T5_BAR_B_FULL + s), 0, ct * T5_TN, 0);
        bw::bulk_load(base + vOff + (uint32_t)s * VBYTES, a.v + (size_t)ct * VF,
                      VBYTES, bar(T5_BAR_B_FULL + s));
        ++issued_b;
      }
      // wait (bounded, quietly) for this lane's own copies: the last one of
      // each stage and of the row operand.  After a normal run all have been
      // consumed and every wait returns at once.
      for (int64_t q = (issued_b > T5_ST ? issued_b - T5_ST : 0); q < issued_b; ++q)
        bw::mbar_wait(bar(T5_BAR_B_FULL + (int)(q % T5_ST)), (uint32_t)((q / T5_ST) & 1),
                      T5_WAIT_BUDGET >> 4);
      if (issued_a > 0)
        bw::mbar_wait(bar(T5_BAR_A_FULL), (uint32_t)((issued_a - 1) & 1), T5_WAIT_BUDGET >> 4);
    }
    __syncwarp();
  } else if (warp == T5_MMA_WARP) {
    // ----------------------------------------------------------------- MMA
    if (lane == 0) {
      constexpr uint32_t IDESC = bw::idesc_f16_f32(T5_TM, T5_TN);
      int64_t kt = 0;
      int seg = 0;
      int ct = ct_first;
      for (int64_t p = p_begin; p < p_end; ++p, ++kt, (++ct == a.C ? ct = 0 : 0)) {
        if (p == p_begin || ct == 0) {
          if (!wait(T5_BAR_A_FULL, (uint32_t)(seg & 1))) break;
          ++seg;
        }
        const int s = (int)(kt % T5_ST);
        const int buf = (int)(kt & 1);
        if (!wait(T5_BAR_B_FULL + s, (uint32_t)((kt / T5_ST) & 1))) break;
        if (!wait(T5_BAR_D_EMPTY + buf, (uint32_t)((kt >> 1) & 1) ^ 1u)) break;
        bw::tc_fence_after();
#pragma unroll
        for (int rt = 0; rt < T5_RT; ++rt) {
          const uint32_t d = tmem + (uint32_t)((buf * T5_RT + rt) * T5_TN);
          const uint32_t aBase = sA + rt * KB * T5_BLK, bBase = sB + s * KB * T5_BLK;
          uint32_t acc = 0;
#pragma unroll
          for (int kc = 0; kc < NH; ++kc) {
            bw::mma_f16(d, bw::sdesc_kmajor_sw32(aBase + (NH + kc) * T5_BLK),
                        bw::sdesc_kmajor_sw32(bBase + kc * T5_BLK), IDESC, acc);
            acc = 1;
            bw::mma_f16(d, bw::sdesc_kmajor_sw32(aBase + kc * T5_BLK),
                        bw::sdesc_kmajor_sw32(bBase + (NH + kc) * T5_BLK), IDESC, 1);
          }
          if (CSEP)
            bw::mma_f16(d, bw::sdesc_kmajor_sw32(aBase + 2 * NH * T5_BLK),
                        bw::sdesc_kmajor_sw32(bBase + 2 * NH * T5_BLK), IDESC, 1);
#pragma unroll
          for (int kc = 0; kc < NH; ++kc)
            bw::mma_f16(d, bw::sdesc_kmajor_sw32(aBase + kc * T5_BLK),
                        bw::sdesc_kmajor_sw32(bBase + kc * T5_BLK), IDESC, 1);
        }
        bw::mma_commit(bar(T5_BAR_D_FULL + buf));
        bw::mma_commit(bar(T5_BAR_B_EMPTY + s));
        if (p + 1 == p_end || ct + 1 == a.C) bw::mma_commit(bar(T5_BAR_A_EMPTY));
      }
      // every MMA issued so far has completed once FIN flips
      if (p_begin < p_end) {
        bw::mma_commit(bar(T5_BAR_FIN));
        bw::mbar_wait(bar(T5_BAR_FIN), 0, T5_WAIT_BUDGET >> 4);
      }
    }
    __syncwarp();
  } else {
    // ------------------------------------------------------------ epilogue
    const int qd = warp & 3;        // TMEM lane quarter
    const int slot = warp >> 2;     // slot of the partial sums
    const int cg = slot % T5_CG;    // column group
    const int tg = slot / T5_CG;    // tiles of this parity (TG = 2)
    constexpr int NBT = T5_WCOLS / 16;   // batches of 16 columns per tile
    if constexpr (TV) {
      const int g = lane >> 2, tq = lane & 3;
      constexpr int NG = T5_RT * 2;      // m16 row groups of a warp: (row tile, half)
      float yacc[NG][NB][4], ytot[TOTF ? 1 : NG][TOTF ? 1 : NB][4];
      float4 *mytot = sTot + warp * (NG * NB) * 32 + lane;   // TOTF: group gr, fragment f at gr NB + f
#pragma unroll
      for (int gr = 0; gr < NG; ++gr)
#pragma unroll
        for (int f = 0; f < NB; ++f)
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            yacc[gr][f][i] = 0.0f;
            if constexpr (!TOTF) ytot[gr][f][i] = 0.0f;
          }
      if constexpr (TOTF > 0) {
#pragma unroll
        for (int q = 0; q < NG * NB; ++q) mytot[q * 32] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
      }
      int64_t kt = 0, rb = rb_first;
      int ct = ct_first;
      // segment end: accumulator (g, 2t + e) / (g + 8, 2t + e) holds B slot 2t + e;
      // add each v_hi slot's v_lo partner and write this warp's partial sums
      // (scaled by 2^14 s_c; t5_reduce_kernel undoes it)
      auto flush = [&](int64_t rbq) {
        const int j = (int)(rbq - rb_first);
        float *out = a.part + (((int64_t)b * a.J + j) * (EW / 4) + slot) * (int64_t)M * T5_RB;
#pragma unroll
        for (int gr = 0; gr < NG; ++gr) {
          float yt[NB][4];   // the totals, cleared as they are read
#pragma unroll
          for (int f = 0; f < NB; ++f) {
            if constexpr (TOTF > 0) {
              float4 &t = mytot[(gr * NB + f) * 32];
              yt[f][0] = t.x, yt[f][1] = t.y, yt[f][2] = t.z, yt[f][3] = t.w;
              t = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
            } else {
#pragma unroll
              for (int i = 0; i < 4; ++i) {
                yt[f][i] = ytot[gr][f][i];
                ytot[gr][f][i] = 0.0f;
              }
            }
          }
          // columns 8 h .. 8 h + 7 of the right-hand sides
#pragma unroll
          for (int h = 0; h < (NB + 1) / 2; ++h) {
            float y[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              if constexpr (NB >= 2)
                y[i] = yt[h][i] + yt[h + NB / 2][i];
              else
                y[i] = yt[0][i] + __shfl_xor_sync(0xffffffffu, yt[0][i], M / 2);
            }
            const int c0 = 8 * h + 2 * tq;
            if (c0 < M) {
              const int row = (gr >> 1) * T5_TM + 32 * qd + 16 * (gr & 1) + g;
              out[c0 * T5_RB + row] = y[0];
              out[(c0 + 1) * T5_RB + row] = y[1];
              out[c0 * T5_RB + row + 8] = y[2];
              out[(c0 + 1) * T5_RB + row + 8] = y[3];
            }
          }
        }
      };
      for (int64_t p = p_begin; p < p_end; ++p, ++kt, (++ct == a.C ? (ct = 0, ++rb) : 0)) {
        const bool segend = p + 1 == p_end || ct + 1 == a.C;
        if (TG == 2 && (int)(kt & 1) != tg) {
          if (segend) flush(rb);
          continue;
        }
        const int s = (int)(kt % T5_ST);
        const int buf = (int)(kt & 1);
        const bool ok = __all_sync(0xffffffffu, wait(T5_BAR_D_FULL + buf, (uint32_t)((kt >> 1) & 1)) &&
                                                    wait(T5_BAR_B_FULL + s, (uint32_t)((kt / T5_ST) & 1)));
        if (!ok) break;
        bw::tc_fence_after();
        const uint2 *vf = reinterpret_cast<const uint2 *>(sV + (size_t)s * VF);
        const uint32_t tcol = tmem + (uint32_t)(buf * T5_RT * T5_TN + cg * T5_WCOLS);
        uint32_t r[PIPE ? 2 : 1][32];   // [batch parity][row group][8]
        auto load_batch = [&](int bt, uint32_t *rr) {
#pragma unroll
          for (int rt = 0; rt < T5_RT; ++rt)
#pragma unroll
            for (int hf = 0; hf < 2; ++hf)
              bw::tmem_ld_16x256b_x2(tcol + ((uint32_t)(32 * qd + 16 * hf) << 16) +
                                         (uint32_t)(rt * T5_TN + bt * 16),
                                     &rr[(rt * 2 + hf) * 8]);
        };
        auto release_buffer = [&]() {
          bw::tc_fence_before();
          __syncwarp();
          if (lane == 0) bw::mbar_arrive(bar(T5_BAR_D_EMPTY + buf));
        };
        if (PIPE) {
          load_batch(0, r[0]);
          bw::tmem_wait_ld32(r[0]);
          if (NBT == 1) release_buffer();
        }
#pragma unroll
        for (int bt = 0; bt < NBT; ++bt) {
          uint32_t *cur = r[PIPE ? (bt & 1) : 0];
          if (PIPE) {
            if (bt + 1 < NBT) load_batch(bt + 1, r[(bt + 1) & 1]);
          } else {
            load_batch(bt, cur);
            bw::tmem_wait_ld32(cur);
            if (bt + 1 == NBT) release_buffer();
          }
          uint2 bf[NB];
#pragma unroll
          for (int f = 0; f < NB; ++f) bf[f] = vf[((cg * NBT + bt) * NB + f) * 32 + lane];
#pragma unroll
          for (int gr = 0; gr < NG; ++gr) {
            // registers (g, 2t), (g, 2t+1), (g+8, 2t), (g+8, 2t+1), then the
            // same for columns 8..15: fragments a0..a3 in order
            const uint32_t *q = &cur[gr * 8];
            uint32_t ah[4], al[4];
#pragma unroll
            for (int pr = 0; pr < 4; ++pr)
              t5_split_pair(t5_kappa_scaled<KERN>(q[2 * pr]), t5_kappa_scaled<KERN>(q[2 * pr + 1]),
                            ah[pr], al[pr]);
#pragma unroll
            for (int f = 0; f < NB; ++f) {
              t5_mma_16816(yacc[gr][f], al, bf[f]);
              t5_mma_16816(yacc[gr][f], ah, bf[f]);
            }
          }
          if (PIPE && bt + 1 < NBT) {
            bw::tmem_wait_ld32(r[(bt + 1) & 1]);
            if (bt + 2 == NBT) release_buffer();
          }
          if ((bt & 3) == 3 || bt + 1 == NBT) {   // sums of 64 columns
#pragma unroll
            for (int gr = 0; gr < NG; ++gr)
#pragma unroll
              for (int f = 0; f < NB; ++f) {
                if constexpr (TOTF > 0) {
                  float4 &t = mytot[(gr * NB + f) * 32];
                  const float4 v = t;
                  t = make_float4(v.x + yacc[gr][f][0], v.y + yacc[gr][f][1], v.z + yacc[gr][f][2],
                                  v.w + yacc[gr][f][3]);
#pragma unroll
                  for (int i = 0; i < 4; ++i) yacc[gr][f][i] = 0.0f;
                } else {
#pragma unroll
                  for (int i = 0; i < 4; ++i) {
                    ytot[gr][f][i] += yacc[gr][f][i];
                    yacc[gr][f][i] = 0.0f;
                  }
                }
              }
          }
        }
        __syncwarp();
        if (lane == 0) bw::mbar_arrive(bar(T5_BAR_V_EMPTY + s));
        if (segend) flush(rb);
      }
    } else {
      // a lane's rows of the two row tiles: packed sums over 32 even and 32 odd
      // columns (acc) and over the segment's finished tiles (tot): two-level
      // float32 accumulation, so a long segment (up to about 1e5 columns per
      // row) adds one sum at a time to its running total instead of one entry at
      // a time.  With up to two right-hand sides, where ex2 leaves the FMA pipe
      // idle (1.75 ms either way at N = 1e5, d = 16; with four 2.30 -> 2.35), the
      // chains are half as long and the tile's sums make a level of their own
      // (mid): a small product's error is its chains'.
      constexpr bool FINE = M == 2 && EW == 16;
      float2 acc[T5_RT][M];
      float mid[T5_RT][FINE ? M : 1], tot[T5_RT][M];
#pragma unroll
      for (int rt = 0; rt < T5_RT; ++rt)
#pragma unroll
        for (int c = 0; c < M; ++c) {
          acc[rt][c] = f2(0.0f, 0.0f);
          if constexpr (FINE) mid[rt][c] = 0.0f;
          tot[rt][c] = 0.0f;
        }
      auto fold = [&](bool last) {
#pragma unroll
        for (int rt = 0; rt < T5_RT; ++rt)
#pragma unroll
          for (int c = 0; c < M; ++c) {
            if constexpr (FINE) {
              mid[rt][c] += acc[rt][c].x + acc[rt][c].y;
              if (last) {
                tot[rt][c] += mid[rt][c];
                mid[rt][c] = 0.0f;
              }
            } else {
              tot[rt][c] += acc[rt][c].x + acc[rt][c].y;
            }
            acc[rt][c] = f2(0.0f, 0.0f);
          }
      };
      // segment end: this warp's partial sums
      auto flush = [&](int64_t rbq) {
        const int j = (int)(rbq - rb_first);
        float *out = a.part + (((int64_t)b * a.J + j) * (EW / 4) + slot) * (int64_t)M * T5_RB +
                     32 * qd + lane;
#pragma unroll
        for (int rt = 0; rt < T5_RT; ++rt)
#pragma unroll
          for (int c = 0; c < M; ++c) {
            out[c * T5_RB + rt * T5_TM] = tot[rt][c];
            tot[rt][c] = 0.0f;
          }
      };
      // kernel values of one batch: [row tile][column pair]
      auto kappa_batch = [&](const uint32_t *cur, float2 *kq) {
#pragma unroll
        for (int i = 0; i < T5_RT * 8; ++i)
          kq[i] = f2(t5_kappa<KERN>(cur[2 * i]), t5_kappa<KERN>(cur[2 * i + 1]));
      };
      auto ffma_batch = [&](const float2 *kq, const float4 *vq) {
#pragma unroll
        for (int jp = 0; jp < 8; ++jp)
#pragma unroll
          for (int cp = 0; cp < MP; ++cp) {
            const float4 v = vq[cp * (T5_TN / 2) + jp];
#pragma unroll
            for (int rt = 0; rt < T5_RT; ++rt) {
              acc[rt][2 * cp] = __ffma2_rn(kq[rt * 8 + jp], f2(v.x, v.y), acc[rt][2 * cp]);
              acc[rt][2 * cp + 1] = __ffma2_rn(kq[rt * 8 + jp], f2(v.z, v.w), acc[rt][2 * cp + 1]);
            }
          }
      };
      // LAG: the batch whose accumulation is pending
      float2 kp[T5_RT * 8];
      const float4 *vp = sV;
      int sp = 0;
      bool havep = false, p_full = false, p_last = false, p_segend = false;
      int64_t p_rb = 0;
      auto retire = [&](const float2 *kq, const float4 *vq, int sq, bool full, bool last,
                        bool segend, int64_t rbq) {
        ffma_batch(kq, vq);
        if (full) fold(last);   // every 32 or 64 columns
        if (last) {
          __syncwarp();
          if (lane == 0) bw::mbar_arrive(bar(T5_BAR_V_EMPTY + sq));
          if (segend) flush(rbq);
        }
      };
      int64_t kt = 0, rb = rb_first;
      int ct = ct_first;
      for (int64_t p = p_begin; p < p_end; ++p, ++kt, (++ct == a.C ? (ct = 0, ++rb) : 0)) {
        const bool segend = (p + 1 == p_end) || (ct + 1 == a.C);
        if (TG == 2 && (int)(kt & 1) != tg) {
          if (segend) {
            if (LAG && havep) retire(kp, vp, sp, p_full, p_last, p_segend, p_rb);
            havep = false;
            flush(rb);
          }
          continue;
        }
        const int s = (int)(kt % T5_ST);
        const int buf = (int)(kt & 1);
        // D of this tile, and (for the visibility of the bulk-copied V) the
        // stage's arrival
        const bool ok =
            __all_sync(0xffffffffu, wait(T5_BAR_D_FULL + buf, (uint32_t)((kt >> 1) & 1)) &&
                                        wait(T5_BAR_B_FULL + s, (uint32_t)((kt / T5_ST) & 1)));
        if (!ok) break;
        bw::tc_fence_after();
        const float4 *vt = sV + (size_t)s * VF + cg * (T5_WCOLS / 2);
        const uint32_t tcol = tmem + ((uint32_t)(32 * qd) << 16) +
                              (uint32_t)(buf * T5_RT * T5_TN + cg * T5_WCOLS);
        // with PIPE, the TMEM loads of batch bt + 1 are in flight while batch bt
        // is computed
        uint32_t r[PIPE ? 2 : 1][32];   // [batch parity][row tile][column]
        auto load_batch = [&](int bt, uint32_t *rr) {
#pragma unroll
          for (int rt = 0; rt < T5_RT; ++rt)
            bw::tmem_ld_32x32b_x16(tcol + (uint32_t)(rt * T5_TN + bt * 16), rr + rt * 16);
        };
        auto release_buffer = [&]() {
          // this warp's TMEM loads of the buffer have landed: hand it back
          bw::tc_fence_before();
          __syncwarp();
          if (lane == 0) bw::mbar_arrive(bar(T5_BAR_D_EMPTY + buf));
        };
        if (PIPE) {
          load_batch(0, r[0]);
          bw::tmem_wait_ld32(r[0]);
          if (NBT == 1) release_buffer();
        }
#pragma unroll
        for (int bt = 0; bt < NBT; ++bt) {
          uint32_t *cur = r[PIPE ? (bt & 1) : 0];
          if (PIPE) {
            if (bt + 1 < NBT) load_batch(bt + 1, r[(bt + 1) & 1]);
          } else {
            load_batch(bt, cur);
            bw::tmem_wait_ld32(cur);
            if (bt + 1 == NBT) release_buffer();
          }
          float2 kc[T5_RT * 8];
          kappa_batch(cur, kc);
          const bool last = bt + 1 == NBT, full = last || (FINE ? bt & 1 : (bt & 3) == 3);
          if constexpr (LAG) {
            if (havep) retire(kp, vp, sp, p_full, p_last, p_segend, p_rb);
          } else {
            retire(kc, vt + bt * 8, s, full, last, segend, rb);
          }
          if (PIPE && bt + 1 < NBT) {
            bw::tmem_wait_ld32(r[(bt + 1) & 1]);
            if (bt + 2 == NBT) release_buffer();
          }
          if constexpr (LAG) {
#pragma unroll
            for (int i = 0; i < T5_RT * 8; ++i) kp[i] = kc[i];
            vp = vt + bt * 8;
            sp = s;
            havep = true;
            p_full = full;
            p_last = last;
            p_segend = last && segend;
            p_rb = rb;
          }
        }
      }
      if (LAG && havep) retire(kp, vp, sp, p_full, p_last, p_segend, p_rb);
    }
  }

  bw::tc_fence_before();
  __syncthreads();
  if (warp == T5_MMA_WARP) {
    bw::tc_fence_after();
    bw::tmem_dealloc(tmem, T5_TMEM_COLS);
  }
}

// CTA whose pair range contains pair p: the largest b with floor(b T / G) <= p.
__host__ __device__ inline int t5_cta_of(int64_t p, int64_t T, int G) {
  return (int)(((p + 1) * (int64_t)G + T - 1) / T) - 1;
}

// Epilogue variants of the tcgen05 product: 1 = 8 warps with pipelined TMEM
// loads, 2 = 16 warps, 3 = 8 warps without the pipelining, 4 = 16 warps with
// it, 5 = 8 warps, pipelined and software-pipelined by one batch, 6 = 12 warps
// on 96-column tiles with pipelined loads, 7 = the same without; 8..11 take
// the sums over V on the tensor cores (TV): 8 = 8 warps with pipelined loads,
// 9 = 8 warps without, 10 = 16 warps without, 11 = 16 warps with.  The 12-
// and 16-warp and software-pipelined variants serve M <= 4 only; M = 16 has
// the TV variants 8 and 9.
constexpr int T5_NVARIANTS = 11;
__host__ __device__ constexpr bool t5_variant_tv(int v) { return v >= 8; }
__host__ __device__ constexpr int t5_variant_ew(int v) {
  return (v == 2 || v == 4 || v == 10 || v == 11) ? 16 : ((v == 6 || v == 7) ? 12 : 8);
}
__host__ __device__ constexpr int t5_variant_tn(int v) { return (v == 6 || v == 7) ? 96 : 128; }
// The tensor-core sums serve square products only: there every row's largest
// kernel value is kappa_ii = 1, while a rectangular product (prediction,
// restricted KRR) may have rows whose kernel values all lie below 2^-20,
// where their fp16 halves (even scaled by 2^14) keep too few bits.
inline bool t5_variant_valid(int v, int M, bool square) {
  return v >= 1 && v <= T5_NVARIANTS &&
         (v == 8 || v == 9 || ((v == 1 || v == 3) && M <= 8) || M <= 4) &&
         (square || !t5_variant_tv(v));
}

// Launches the instance for (nh, csep, M, variant); cudaErrorInvalidValue for
// a shape without one.  Defined per kernel function and family (TV or not) in
// kmvtc5_gauss.cu, kmvtc5_matern.cu, kmvtc5_tv_gauss.cu, kmvtc5_tv_matern.cu.
cudaError_t launch_kmvtc5_gauss(int nh, int csep, int M, int variant, int G, size_t smem,
                                cudaStream_t s, const CUtensorMap &rowmap,
                                const CUtensorMap &colmap, const T5Args &a);
cudaError_t launch_kmvtc5_matern(int nh, int csep, int M, int variant, int G, size_t smem,
                                 cudaStream_t s, const CUtensorMap &rowmap,
                                 const CUtensorMap &colmap, const T5Args &a);
cudaError_t launch_kmvtc5_tv_gauss(int nh, int csep, int M, int variant, int G, size_t smem,
                                   cudaStream_t s, const CUtensorMap &rowmap,
                                   const CUtensorMap &colmap, const T5Args &a);
cudaError_t launch_kmvtc5_tv_matern(int nh, int csep, int M, int variant, int G, size_t smem,
                                    cudaStream_t s, const CUtensorMap &rowmap,
                                    const CUtensorMap &colmap, const T5Args &a);

template <int KERN, int NH, int CS, int M, int EW, int PIPE, int LAG = 0, int TN = 128, int TV = 0>
cudaError_t launch_kmvtc5_one(int G, size_t smem, cudaStream_t s, const CUtensorMap &rowmap,
                              const CUtensorMap &colmap, const T5Args &a) {
  auto k = kmvtc5_kernel<KERN, NH, CS, M, EW, PIPE, LAG, TN, TV>;
  if (raise_smem_limit(k, smem) != KRR_OK) return cudaErrorInvalidValue;
  k<<<G, (EW + 2) * 32, smem, s>>>(rowmap, colmap, a);
  return cudaGetLastError();
}

template <int KERN, int NH, int CS, int M, bool TVSET>
cudaError_t launch_kmvtc5_m(int variant, int G, size_t smem, cudaStream_t s,
                            const CUtensorMap &rowmap, const CUtensorMap &colmap,
                            const T5Args &a) {
  if constexpr (TVSET) {
    switch (variant) {
      case 8: return launch_kmvtc5_one<KERN, NH, CS, M, 8, 1, 0, 128, 1>(G, smem, s, rowmap, colmap, a);
      case 9: return launch_kmvtc5_one<KERN, NH, CS, M, 8, 0, 0, 128, 1>(G, smem, s, rowmap, colmap, a);
      case 10:
        if constexpr (M <= 4) return launch_kmvtc5_one<KERN, NH, CS, M, 16, 0, 0, 128, 1>(G, smem, s, rowmap, colmap, a);
        break;
      case 11:
        if constexpr (M <= 4) return launch_kmvtc5_one<KERN, NH, CS, M, 16, 1, 0, 128, 1>(G, smem, s, rowmap, colmap, a);
        break;
    }
  } else {
    switch (variant) {
      case 1: return launch_kmvtc5_one<KERN, NH, CS, M, 8, 1>(G, smem, s, rowmap, colmap, a);
      case 3: return launch_kmvtc5_one<KERN, NH, CS, M, 8, 0>(G, smem, s, rowmap, colmap, a);
      case 2:
        if constexpr (M <= 4) return launch_kmvtc5_one<KERN, NH, CS, M, 16, 0>(G, smem, s, rowmap, colmap, a);
        break;
      case 4:
        if constexpr (M <= 4) return launch_kmvtc5_one<KERN, NH, CS, M, 16, 1>(G, smem, s, rowmap, colmap, a);
        break;
      case 5:
        if constexpr (M <= 4) return launch_kmvtc5_one<KERN, NH, CS, M, 8, 1, 1>(G, smem, s, rowmap, colmap, a);
        break;
      case 6:
        if constexpr (M <= 4) return launch_kmvtc5_one<KERN, NH, CS, M, 12, 1, 0, 96>(G, smem, s, rowmap, colmap, a);
        break;
      case 7:
        if constexpr (M <= 4) return launch_kmvtc5_one<KERN, NH, CS, M, 12, 0, 0, 96>(G, smem, s, rowmap, colmap, a);
        break;
    }
  }
  return cudaErrorInvalidValue;
}

template <int KERN, bool TVSET>
cudaError_t launch_kmvtc5(int nh, int csep, int M, int variant, int G, size_t smem,
                          cudaStream_t s, const CUtensorMap &rowmap, const CUtensorMap &colmap,
                          const T5Args &a) {
#define KRR_T5_CASE(NH, CS, MM)                                                         \
  if (nh == NH && csep == CS && M == MM)                                              \
    return launch_kmvtc5_m<KERN, NH, CS, MM, TVSET>(variant, G, smem, s, rowmap, colmap, a);
  KRR_T5_CASE(1, 0, 2) KRR_T5_CASE(1, 0, 4) KRR_T5_CASE(1, 0, 8)
  KRR_T5_CASE(1, 1, 2) KRR_T5_CASE(1, 1, 4) KRR_T5_CASE(1, 1, 8)
  KRR_T5_CASE(2, 0, 2) KRR_T5_CASE(2, 0, 4) KRR_T5_CASE(2, 0, 8)
  KRR_T5_CASE(2, 1, 2) KRR_T5_CASE(2, 1, 4) KRR_T5_CASE(2, 1, 8)
  if constexpr (TVSET) {
    KRR_T5_CASE(1, 0, 16) KRR_T5_CASE(1, 1, 16) KRR_T5_CASE(2, 0, 16) KRR_T5_CASE(2, 1, 16)
  }
#undef KRR_T5_CASE
  return cudaErrorInvalidValue;
}

}  // namespace krr
