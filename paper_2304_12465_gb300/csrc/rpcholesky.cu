// Blocked RPCholesky (Alg. 3) on the device, float64.
//
// Per block: (1) fixed-point pivot sampling from the residual diagonal
// (residuals at or below the drop threshold carry no weight) and
// Unique in first-occurrence order; (2) G = A(:,S') from the kernel function
// minus the Schur term F(:,1:i) F(S',1:i)^T (by digits on the tensor cores);
// (3) Cholesky of G(S',S') pivot by pivot with the drop rule; (4) the new
// columns G R^{-1}, by groups of columns: the groups before them on the tensor
// cores, then forward substitution, fused with the residual-diagonal downdate.
#include <algorithm>

#include "dense.cuh"
#include "handles.cuh"
#include "kmv.cuh"
#include "rpc.cuh"

namespace krr {

// ------------------------------------------------------------- sampler
__device__ __forceinline__ uint64_t fixed_weight(double v, double dfloor, int fbits) {
  if (!(v > 0.0) || !(v > dfloor)) return 0ull;
  if (v > 1.0) v = 1.0;
  return __double2ull_rz(ldexp(v, fbits));
}

int fixed_point_bits(int64_t N) {
  int c = 0;
  while (((int64_t)1 << c) < N) ++c;
  return 62 - c;
}

constexpr int SMP_THREADS = 256;
constexpr int SMP_MAX_CHUNKS = 4096;

static int64_t sampler_chunk(int64_t N) {
  int64_t ch = 2048;
  while ((N + ch - 1) / ch > SMP_MAX_CHUNKS) ch *= 2;
  return ch;
}

__global__ void __launch_bounds__(SMP_THREADS)
sample_chunk_sums_kernel(const double *__restrict__ dres, int64_t N, double dfloor,
                         int fbits, int64_t chunk, uint64_t *__restrict__ csum) {
  __shared__ uint64_t red[SMP_THREADS / 32];
  const int64_t b0 = (int64_t)blockIdx.x * chunk;
  const int64_t b1 = min(N, b0 + chunk);
  uint64_t s = 0;
  for (int64_t i = b0 + threadIdx.x; i < b1; i += SMP_THREADS) s += fixed_weight(dres[i], dfloor, fbits);
  s = warp_sum(s);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    uint64_t t = 0;
    for (int w = 0; w < SMP_THREADS / 32; ++w) t += red[w];
    csum[blockIdx.x] = t;
  }
}

// Exclusive prefix of v over the block's threads, and the block's total.
__device__ __forceinline__ uint64_t block_scan_u64(uint64_t v, uint64_t *total,
                                                   uint64_t (&warp_sums)[SMP_THREADS / 32]) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint64_t incl = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint64_t u = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += u;
  }
  __syncthreads();   // a previous scan's sums have been read
  if (lane == 31) warp_sums[warp] = incl;
  __syncthreads();
  uint64_t before = 0, all = 0;
#pragma unroll
  for (int w = 0; w < SMP_THREADS / 32; ++w) {
    if (w < warp) before += warp_sums[w];
    all += warp_sums[w];
  }
  *total = all;
  return before + incl - v;
}

// One CTA a draw: the chunk that holds the target (from the chunk sums), then
// the entry inside it, each by a block-wide prefix over consecutive shares.
// One CTA for all draws took 490 us for 100 draws at N = 1e5 (a chunk's scan
// by one warp, thirteen draws a warp, the chunk sums by one thread).
// counts[0] = ndraw, or 0 when every weight is zero.
__global__ void __launch_bounds__(SMP_THREADS)
sample_draw_kernel(const double *__restrict__ dres, int64_t N, double dfloor, int fbits,
                   int64_t chunk, const uint64_t *__restrict__ csum, int nchunks, uint64_t seed,
                   uint64_t t, int ndraw, int64_t *__restrict__ draws, int *__restrict__ counts) {
  __shared__ uint64_t ws[SMP_THREADS / 32];
  __shared__ uint64_t s_local;
  __shared__ int s_chunk;
  const int tid = threadIdx.x, j = blockIdx.x;
  const int per = (nchunks + SMP_THREADS - 1) / SMP_THREADS;
  const int c0 = min(nchunks, tid * per), c1 = min(nchunks, c0 + per);
  uint64_t mine = 0, total;
  for (int c = c0; c < c1; ++c) mine += csum[c];
  uint64_t run = block_scan_u64(mine, &total, ws);
  if (j == 0 && tid == 0) counts[0] = total ? ndraw : 0;
  if (total == 0) return;
  uint64_t ctr[4] = {t, (uint64_t)j, 0ull, 0ull}, out[4];
  philox4x64_10(ctr, seed, kTagPivots, out);
  const uint64_t target = scale_u64(out[0], total);
  // smallest chunk whose inclusive prefix exceeds the target
  if (target >= run && target < run + mine) {
    int c = c0;
    while (target >= run + csum[c]) run += csum[c++];
    s_chunk = c;
    s_local = target - run;
  }
  __syncthreads();
  uint64_t tl = s_local;
  const int64_t b1 = min(N, (int64_t)(s_chunk + 1) * chunk);
  constexpr int PER = 8;
  for (int64_t b0 = (int64_t)s_chunk * chunk; b0 < b1; b0 += SMP_THREADS * PER) {
    const int64_t i0 = b0 + (int64_t)tid * PER;
    uint64_t w[PER];
    mine = 0;
#pragma unroll
    for (int e = 0; e < PER; ++e) {
      w[e] = (i0 + e < b1) ? fixed_weight(dres[i0 + e], dfloor, fbits) : 0ull;
      mine += w[e];
    }
    uint64_t part;
    run = block_scan_u64(mine, &part, ws);
    if (tl < part) {
      if (tl >= run && tl < run + mine) {
        int e = 0;
        while (tl >= run + w[e]) run += w[e++];
        draws[j] = i0 + e;
      }
      return;
    }
    tl -= part;
  }
}

// Unique: the distinct draws in first-occurrence order; one thread a draw.
constexpr int UNIQUE_THREADS = 1024;
__global__ void __launch_bounds__(UNIQUE_THREADS)
sample_unique_kernel(const int64_t *__restrict__ draws, int64_t *__restrict__ cand,
                     int *__restrict__ counts) {
  __shared__ int64_t sd[UNIQUE_THREADS];
  __shared__ int wsum[UNIQUE_THREADS / 32];
  const int j = threadIdx.x, lane = j & 31, warp = j >> 5, n = counts[0];
  if (n == 0) {
    if (j == 0) counts[1] = 0;
    return;
  }
  const int64_t v = j < n ? draws[j] : -1;
  sd[j] = v;
  __syncthreads();
  bool first = j < n;
  for (int i = 0; i < j && first; ++i) first = sd[i] != v;
  const unsigned b = __ballot_sync(0xffffffffu, first);
  if (lane == 0) wsum[warp] = __popc(b);
  __syncthreads();
  int pos = __popc(b & ((1u << lane) - 1u)), all = 0;
  for (int w = 0; w < (int)(blockDim.x >> 5); ++w) {
    if (w < warp) pos += wsum[w];
    all += wsum[w];
  }
  if (first) cand[pos] = v;
  if (j == 0) counts[1] = all;
}

krr_status rpc_sample_device(const double *dres, int64_t N, double dfloor, uint64_t seed,
                             uint64_t t, int ndraw, int64_t *draws, int64_t *cand, int *counts,
                             cudaStream_t s) {
  const int fbits = fixed_point_bits(N);
  const int64_t chunk = sampler_chunk(N);
  const int nchunks = (int)((N + chunk - 1) / chunk);
  DevBuf<uint64_t> csum;
  KRR_TRY(csum.alloc(nchunks, s));
  sample_chunk_sums_kernel<<<nchunks, SMP_THREADS, 0, s>>>(dres, N, dfloor, fbits, chunk,
                                                           csum.p);
  KRR_LAUNCH_CHECK();
  sample_draw_kernel<<<ndraw, SMP_THREADS, 0, s>>>(dres, N, dfloor, fbits, chunk, csum.p, nchunks,
                                                   seed, t, ndraw, draws, counts);
  KRR_LAUNCH_CHECK();
  sample_unique_kernel<<<1, (ndraw + 31) / 32 * 32, 0, s>>>(draws, cand, counts);
  KRR_LAUNCH_CHECK();
  return KRR_OK;
}

// --------------------------------------------- uniform and greedy rules
// The pivot rules the paper compares RPCholesky with (Sec. 4).
//
// Uniform: a uniformly random k-subset of the columns, drawn independently
// of A: draw q takes word 0 of Philox(counter (q, 0, 1, 0), key (seed, pivot
// tag)) as floor(u N / 2^64), keeping first occurrences (a bitmap of the
// columns seen) until k distinct indices are found.  One thread; the loop is
// bounded (far above the expected k + k^2 / (2N) draws for k <= N) and
// reports failure through out_count.
__global__ void uniform_pivots_kernel(int64_t N, int k, uint64_t seed, unsigned *__restrict__ seen,
                                      int64_t *__restrict__ S, int *__restrict__ out_count) {
  if (threadIdx.x != 0 || blockIdx.x != 0) return;
  int got = 0;
  const uint64_t qmax = 64ull * (uint64_t)k + 4096ull;
  for (uint64_t q = 0; got < k && q < qmax; ++q) {
    uint64_t ctr[4] = {q, 0ull, 1ull, 0ull}, out[4];
    philox4x64_10(ctr, seed, kTagPivots, out);
    const int64_t i = (int64_t)scale_u64(out[0], (uint64_t)N);
    const unsigned bit = 1u << (i & 31);
    if (seen[i >> 5] & bit) continue;
    seen[i >> 5] |= bit;
    S[got++] = i;
  }
  *out_count = got;
}

// Greedy: the npick largest residuals above dfloor in descending order (ties:
// the smallest index); npick = 1 is the paper's rule.  One CTA; pick j is the
// largest (value, -index) strictly below pick j - 1 in that order.
constexpr int GREEDY_THREADS = 1024;

__global__ void __launch_bounds__(GREEDY_THREADS)
greedy_pick_kernel(const double *__restrict__ dres, int64_t N, double dfloor, int npick,
                   int64_t *__restrict__ cand, int *__restrict__ counts) {
  __shared__ double sv[GREEDY_THREADS / 32];
  __shared__ int64_t si[GREEDY_THREADS / 32];
  __shared__ double prev_v;
  __shared__ int64_t prev_i;
  __shared__ int got;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (threadIdx.x == 0) {
    prev_v = INFINITY;
    prev_i = -1;
    got = 0;
  }
  __syncthreads();
  for (int j = 0; j < npick; ++j) {
    const double pv = prev_v;
    const int64_t pi = prev_i;
    double bv = -1.0;
    int64_t bi = -1;
    for (int64_t i = threadIdx.x; i < N; i += GREEDY_THREADS) {
      const double v = dres[i];
      if (!(v > 0.0) || !(v > dfloor)) continue;
      // strictly after the previous pick in (value desc, index asc) order
      if (v > pv || (v == pv && i <= pi)) continue;
      if (bi < 0 || v > bv) {
        bv = v;
        bi = i;
      }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const double ov = __shfl_xor_sync(0xffffffffu, bv, o);
      const int64_t oi = __shfl_xor_sync(0xffffffffu, bi, o);
      if (oi >= 0 && (bi < 0 || ov > bv || (ov == bv && oi < bi))) {
        bv = ov;
        bi = oi;
      }
    }
    if (lane == 0) {
      sv[warp] = bv;
      si[warp] = bi;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      double v = -1.0;
      int64_t b = -1;
      for (int w = 0; w < GREEDY_THREADS / 32; ++w) {
        if (si[w] >= 0 && (b < 0 || sv[w] > v || (sv[w] == v && si[w] < b))) {
          v = sv[w];
          b = si[w];
        }
      }
      if (b >= 0) {
        cand[got] = b;
        got = got + 1;
        prev_v = v;
        prev_i = b;
      }
    }
    __syncthreads();
    if (got <= j) break;   // nothing eligible left
  }
  if (threadIdx.x == 0) {
    counts[0] = got > 0 ? npick : 0;
    counts[1] = got;
  }
}

// ------------------------------------------------------- block kernels
// q = x / d with r = 1 / d at hand: one correction of x r, which leaves the
// rounding of a division at a quarter of its float64 operations.
__device__ __forceinline__ double div_by(double x, double d, double r) {
  const double q = x * r;
  return fma(fma(-q, d, x), r, q);
}

// Right-looking Cholesky of T = G(S', S') (nc x nc) in candidate order; a
// candidate whose current Schur value is <= thr is dropped and does not
// update the rest.  Outputs the factor of the kept candidates Lb (ld nc,
// column-major, lower, in their order), their positions, and their count.
// Panels of eight columns are factored in registers by up to four warps, one
// for each float64 pipe of the SM: a lane keeps one row below the panel's
// diagonal block, and every warp the block itself, so that they need no
// barriers; the rest is updated by all warps between two barriers.  100
// candidates took 262 us with three barriers a column, 231 us with the panel in
// one warp, whose 272 float64 instructions a panel take 67 clocks each, now
// 187.  n2[a]: squared norm of row a of Lb over the columns before its group of
// the triangular solve (trsm_group_start).
constexpr int TRSM_W = 20;   // columns of a group at most, see block_trsm_kernel
__host__ __device__ inline int trsm_groups(int na) { return (na + TRSM_W - 1) / TRSM_W; }
__host__ __device__ inline int trsm_group_start(int na, int q) {
  return na * q / trsm_groups(na);   // na <= 128
}
constexpr int CHOL_PW = 8;
__global__ void __launch_bounds__(256)
block_chol_kernel(const double *__restrict__ G, int64_t ldg, const int64_t *__restrict__ cand,
                  int nc, double thr, double *__restrict__ Lb, int *__restrict__ kept,
                  int *__restrict__ nkept, double *__restrict__ n2) {
  extern __shared__ double sT[];  // nc x (nc + 1), row-major
  __shared__ int s_list[RPC_MAX_BLOCK];
  __shared__ unsigned s_mask;     // kept columns of the panel
  __shared__ int s_na;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int ld = nc + 1;
  for (int e = tid; e < nc * nc; e += blockDim.x) {
    const int c = e / nc, a = e - c * nc;
    sT[a * ld + c] = G[cand[a] + (int64_t)c * ldg];
  }
  if (tid == 0) s_na = 0;
  __syncthreads();
  for (int c0 = 0; c0 < nc; c0 += CHOL_PW) {
    const int pw = min(CHOL_PW, nc - c0);
    double top[CHOL_PW];   // warp 0: the diagonal block, stored once every warp has read it
    const int a = c0 + CHOL_PW + 32 * warp + lane;   // this lane's row below the diagonal block
    if (warp == 0 || (warp < 4 && c0 + CHOL_PW + 32 * warp < nc)) {
      // rows c0 .. c0 + 7 in lanes 0..7 of every warp (T), rows below (P);
      // columns c0 .. c0 + pw
      double T[CHOL_PW], P[CHOL_PW];
#pragma unroll
      for (int q = 0; q < CHOL_PW; ++q) {
        T[q] = (lane < pw && q < pw) ? sT[(c0 + lane) * ld + c0 + q] : 0.0;
        P[q] = (a < nc && q < pw) ? sT[a * ld + c0 + q] : 0.0;
      }
      unsigned mask = 0;
#pragma unroll
      for (int q = 0; q < CHOL_PW; ++q) {
        const double p = __shfl_sync(0xffffffffu, T[q], q);
        if (q < pw && p > thr) {
          mask |= 1u << q;
          double d, rd;
          sqrt_and_inverse(p, &d, &rd);
          T[q] = div_by(T[q], d, rd);
          P[q] = div_by(P[q], d, rd);
          if (lane == q) T[q] = d;
#pragma unroll
          for (int u = q + 1; u < CHOL_PW; ++u) {
            const double l = __shfl_sync(0xffffffffu, T[q], u);
            T[u] = fma(-T[q], l, T[u]);
            P[u] = fma(-P[q], l, P[u]);
          }
        }
      }
#pragma unroll
      for (int q = 0; q < CHOL_PW; ++q) {
        if (a < nc && q < pw) sT[a * ld + c0 + q] = P[q];
        top[q] = T[q];
      }
      if (tid == 0) {
        s_mask = mask;
        int na = s_na;
        for (int q = 0; q < pw; ++q)
          if (mask >> q & 1) s_list[na++] = c0 + q;
        s_na = na;
      }
    }
    __syncthreads();
    if (warp == 0 && lane < pw) {
#pragma unroll
      for (int q = 0; q < CHOL_PW; ++q)
        if (q < pw) sT[(c0 + lane) * ld + c0 + q] = top[q];
    }
    const unsigned mask = s_mask;
    const int t0 = c0 + pw;
    // 16 x 16 threads over the lower triangle that is left
    for (int a = t0 + (tid >> 4); a < nc; a += 16) {
      double x[CHOL_PW];
#pragma unroll
      for (int q = 0; q < CHOL_PW; ++q) x[q] = (mask >> q & 1) ? sT[a * ld + c0 + q] : 0.0;
      for (int b = t0 + (tid & 15); b <= a; b += 16) {
        double v = sT[a * ld + b];
#pragma unroll
        for (int q = 0; q < CHOL_PW; ++q)
          if (mask >> q & 1) v = fma(-x[q], sT[b * ld + c0 + q], v);
        sT[a * ld + b] = v;
      }
    }
    __syncthreads();
  }
  const int na = s_na;
  for (int e = tid; e < na * na; e += blockDim.x) {
    const int c = e / na, a = e - c * na;
    Lb[a + (int64_t)c * nc] = (a >= c) ? sT[s_list[a] * ld + s_list[c]] : 0.0;
  }
  for (int e = tid; e < na; e += blockDim.x) kept[e] = s_list[e];
  {
    // two threads a row (256 threads, at most 128 rows)
    const int e = tid >> 1;
    double v = 0.0;
    if (e < na) {
      int a0 = 0;
      for (int q = 1; trsm_group_start(na, q) <= e; ++q) a0 = trsm_group_start(na, q);
      const double *row = sT + s_list[e] * ld;
#pragma unroll 8
      for (int c = tid & 1; c < a0; c += 2) {
        const double x = row[s_list[c]];
        v = fma(x, x, v);
      }
    }
    v += __shfl_xor_sync(0xffffffffu, v, 1);
    if (e < na && (tid & 1) == 0) n2[e] = v;
  }
  if (tid == 0) *nkept = na;
}

// Columns a0 .. a0 + w of the new part of F: row n solves x L^T = G(n, kept)
// over them by forward substitution (G already holds the part of the columns
// before a0) and writes x to F(n, rank + a0 ..); dres(n) -= |x|^2.  rn2 and bn2
// collect |x|^2 over all columns and over this block's, the scales of the products
// by digits.  The row stays in registers, so a group is at most TRSM_W columns:
// the float64 work of a row is w^2 / 2 + 4 w of the na^2 / 2 + 10 na that
// substitution over all na columns (with divisions) took.
constexpr int TRSM_THREADS = 64;
__global__ void __launch_bounds__(TRSM_THREADS)
block_trsm_kernel(const double *__restrict__ G, int64_t ldg, const double *__restrict__ Lb,
                  int nc, const int *__restrict__ kept, int a0, int w, double *__restrict__ F,
                  int64_t N, int rank, double *__restrict__ dres, double *__restrict__ rn2,
                  double *__restrict__ bn2) {
  __shared__ double sL[TRSM_W][TRSM_W + 1];
  __shared__ double sR[TRSM_W];
  for (int e = threadIdx.x; e < w * w; e += TRSM_THREADS) {
    const int a = e / w, b = e % w;
    const double v = Lb[a0 + a + (int64_t)(a0 + b) * nc];
    sL[a][b] = v;
    if (a == b) sR[a] = 1.0 / v;
  }
  __syncthreads();
  const int64_t n = (int64_t)blockIdx.x * TRSM_THREADS + threadIdx.x;
  if (n >= N) return;
  double x[TRSM_W];
#pragma unroll
  for (int a = 0; a < TRSM_W; ++a) x[a] = a < w ? G[n + (int64_t)kept[a0 + a] * ldg] : 0.0;
  double s2 = 0.0;
  double *Fn = F + n + (int64_t)(rank + a0) * N;
#pragma unroll
  for (int a = 0; a < TRSM_W; ++a) {
    if (a < w) {
      const double v = div_by(x[a], sL[a][a], sR[a]);
      Fn[(int64_t)a * N] = v;
      s2 = fma(v, v, s2);
#pragma unroll
      for (int b = a + 1; b < TRSM_W; ++b)
        if (b < w) x[b] = fma(-v, sL[b][a], x[b]);
    }
  }
  dres[n] -= s2;
  rn2[n] += s2;
  bn2[n] = a0 == 0 ? s2 : bn2[n] + s2;
}

__global__ void block_finish_kernel(const int64_t *__restrict__ cand, int nc,
                                    const int *__restrict__ kept, const int *__restrict__ nkept,
                                    int64_t *__restrict__ S, int rank,
                                    double *__restrict__ dres) {
  const int na = *nkept;
  for (int e = threadIdx.x; e < na; e += blockDim.x) S[rank + e] = cand[kept[e]];
  for (int c = threadIdx.x; c < nc; c += blockDim.x) dres[cand[c]] = 0.0;
}

__global__ void max_reduce_kernel(const double *__restrict__ v, int64_t n,
                                  double *__restrict__ out) {
  __shared__ double red[32];
  double m = 0.0;
  for (int64_t i = threadIdx.x; i < n; i += blockDim.x) m = fmax(m, v[i]);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
  __syncthreads();
  if (threadIdx.x == 0) {
    double r = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) r = fmax(r, red[w]);
    *out = r;
  }
}

// ----------------------------------------------------------- driver
krr_status rpcholesky_device(const double *Xd, int64_t N, int d, int kern, double sigma,
                             int k, int B, uint64_t seed, cudaStream_t s, krr_factor *f,
                             int rule) {
  f->N = N;
  f->d = d;
  f->kern = kern;
  f->sigma = sigma;
  f->k = k;
  f->seed = seed;
  KRR_TRY(dev_alloc(&f->F, (size_t)N * k));
  KRR_TRY(dev_alloc(&f->S, (size_t)k));
  KRR_TRY(dev_alloc(&f->dres, (size_t)N));
  KRR_CUDA_TRY(cudaMemsetAsync(f->F, 0, sizeof(double) * (size_t)N * k, s));
  KRR_TRY(kernel_diag_f64(Xd, N, d, kern, sigma, f->dres, s));

  DevBuf<double> maxd;
  KRR_TRY(maxd.alloc(1, s));
  max_reduce_kernel<<<1, 1024, 0, s>>>(f->dres, N, maxd.p);
  KRR_LAUNCH_CHECK();
  double maxdiag = 0.0;
  KRR_CUDA_TRY(cudaMemcpyAsync(&maxdiag, maxd.p, sizeof(double), cudaMemcpyDeviceToHost, s));
  PointsF64 P64;   // waits for s
  KRR_TRY(prepare_points_f64(Xd, N, d, kern, sigma, s, P64, true));
  const double thr = (double)N * 2.220446049250313e-16 * maxdiag;

  DevBuf<int64_t> draws, cand;
  DevBuf<int> counts, kept;
  DevBuf<double> G, Lb, rn2, bn2, ln2;   // (squared row norms of F, its new block and Lb)
  DevBuf<uint8_t> img;
  KRR_TRY(draws.alloc(B, s));
  KRR_TRY(cand.alloc(B, s));
  KRR_TRY(counts.alloc(4, s));
  KRR_TRY(kept.alloc(B, s));
  KRR_TRY(G.alloc((size_t)N * B, s));
  KRR_TRY(img.alloc(dig_image_bytes(B, std::max(k, B)), s));
  KRR_TRY(Lb.alloc((size_t)B * B, s));
  KRR_TRY(rn2.alloc((size_t)N, s));
  KRR_TRY(bn2.alloc((size_t)N, s));
  KRR_TRY(ln2.alloc((size_t)B, s));
  KRR_CUDA_TRY(cudaMemsetAsync(rn2.p, 0, sizeof(double) * (size_t)N, s));

  KRR_TRY(raise_smem_limit(block_chol_kernel, (size_t)B * (B + 1) * sizeof(double)));

  // the uniform rule's k pivots are drawn before the first block
  DevBuf<int64_t> upiv;
  int nupiv = 0, used = 0;
  if (rule == KRR_PIVOT_UNIFORM) {
    DevBuf<unsigned> seen;
    KRR_TRY(seen.alloc((size_t)(N + 31) / 32, s));
    KRR_TRY(upiv.alloc(k, s));
    KRR_CUDA_TRY(cudaMemsetAsync(seen.p, 0, sizeof(unsigned) * (size_t)((N + 31) / 32), s));
    uniform_pivots_kernel<<<1, 32, 0, s>>>(N, k, seed, seen.p, upiv.p, counts.p);
    KRR_LAUNCH_CHECK();
    KRR_CUDA_TRY(cudaMemcpyAsync(&nupiv, counts.p, sizeof(int), cudaMemcpyDeviceToHost, s));
    KRR_CUDA_TRY(cudaStreamSynchronize(s));
    if (nupiv < k) {
      set_error("uniform pivot draw ended early (%d of %d)", nupiv, k);
      return KRR_ECUDA;
    }
  }

  int rank = 0;
  uint64_t t = 0;
  int hcounts[4];
  while (rule == KRR_PIVOT_UNIFORM ? used < nupiv : rank < k) {
    int nc;
    if (rule == KRR_PIVOT_UNIFORM) {
      nc = (nupiv - used < B) ? (nupiv - used) : B;
      KRR_CUDA_TRY(cudaMemcpyAsync(cand.p, upiv.p + used, sizeof(int64_t) * nc,
                                   cudaMemcpyDeviceToDevice, s));
      used += nc;
      ++t;
    } else {
      const int nd = (k - rank < B) ? (k - rank) : B;
      if (rule == KRR_PIVOT_GREEDY) {
        greedy_pick_kernel<<<1, GREEDY_THREADS, 0, s>>>(f->dres, N, thr, nd, cand.p, counts.p);
        KRR_LAUNCH_CHECK();
      } else {
        KRR_TRY(rpc_sample_device(f->dres, N, thr, seed, t, nd, draws.p, cand.p, counts.p, s));
      }
      ++t;
      KRR_CUDA_TRY(cudaMemcpyAsync(hcounts, counts.p, 2 * sizeof(int), cudaMemcpyDeviceToHost,
                                   s));
      KRR_CUDA_TRY(cudaStreamSynchronize(s));
      if (hcounts[0] == 0) break;
      nc = hcounts[1];
    }
    // G = A(:, S') - F(:, 0:rank) F(S', 0:rank)^T
    KRR_TRY(kernel_columns_f64(P64, cand.p, nc, G.p, N, s));
    if (rank > 0)
      KRR_TRY(dig_gemm_sub(f->F, N, N, rank, rn2.p, f->F, N, cand.p, rn2.p, nc, G.p, N, nullptr,
                           reinterpret_cast<uint4 *>(img.p), s));
    block_chol_kernel<<<1, 256, (size_t)nc * (nc + 1) * sizeof(double), s>>>(
        G.p, N, cand.p, nc, thr, Lb.p, kept.p, counts.p + 2, ln2.p);
    KRR_LAUNCH_CHECK();
    int na = 0;
    KRR_CUDA_TRY(cudaMemcpyAsync(&na, counts.p + 2, sizeof(int), cudaMemcpyDeviceToHost, s));
    KRR_CUDA_TRY(cudaStreamSynchronize(s));
    // equal groups of at most TRSM_W columns
    for (int q = 0; q < trsm_groups(na); ++q) {
      const int a0 = trsm_group_start(na, q), w = trsm_group_start(na, q + 1) - a0;
      KRR_TRY(dig_gemm_sub(f->F + (int64_t)rank * N, N, N, a0, bn2.p, Lb.p + a0, nc, nullptr,
                           ln2.p + a0, w, G.p, N, kept.p + a0, reinterpret_cast<uint4 *>(img.p),
                           s));
      block_trsm_kernel<<<ceil_div(N, TRSM_THREADS), TRSM_THREADS, 0, s>>>(
          G.p, N, Lb.p, nc, kept.p, a0, w, f->F, N, rank, f->dres, rn2.p, bn2.p);
      KRR_LAUNCH_CHECK();
    }
    block_finish_kernel<<<1, 128, 0, s>>>(cand.p, nc, kept.p, counts.p + 2, f->S, rank, f->dres);
    KRR_LAUNCH_CHECK();
    rank += na;
  }
  KRR_TRY(tc5_check_fault(s));   // the digit products' bounded waits
  f->rank = rank;
  f->nblocks = (int)t;
  return KRR_OK;
}

}  // namespace krr
