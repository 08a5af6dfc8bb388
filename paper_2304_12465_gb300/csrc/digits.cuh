// Float64 products of matrices whose rows have norm 1 at most, on the fp16
// tensor cores, by digits (an Ozaki-style splitting).
//
// Every entry is rounded once to the fixed-point integer v = round(2^56 x) and
// written as seven balanced base-256 digits, x = sum_s q_s 2^(-8 - 8 s),
// -128 <= q_s <= 127 (the leading one -512..511, for |x| below 2).  Digits are
// exact in fp16; the product of digits s and t carries 2^(-16 - 8 (s + t)), so
// the pairs of one g = s + t share an accumulator.  Over 128 terms a pair of
// full digits stays within 2^21 and a pair with a leading digit within 128 256
// sqrt(128) (the rows' norm), so seven pairs stay below 2^24 and the float32
// accumulation is exact.  The 28 pairs with s + t <= 6 are kept; what is
// dropped is about 2^-59.6 sqrt(6 K) of 1, below the rounding of a float64 sum
// of K terms.  After 128 terms the seven accumulators go into one 64-bit total
// in units of 2^-60.
//
// One 16 x 8 x 16 MMA does 2048 multiply-adds; the float64 pipe does 1.9 a
// clock and SM, so 28 MMAs (59.6 clocks at the measured rate of 606 TFLOP/s)
// replace 1078 clocks of DFMA, and the float-float form on the float32 pipe
// (12 operations a multiply-add) 192.
#pragma once

#include <cuda_fp16.h>

#include "common.cuh"

namespace krr {

constexpr int DIG_N = 7;              // digits
constexpr int DIG_CHUNK = 128;        // terms between flushes of the accumulators
constexpr int DIG_MAX_COLS = 112;     // columns of one launch

// round(2^56 x), |x| < 2; 0 for |x| < 2^-57.
__device__ __forceinline__ int64_t dig_fixed(double x) {
  const uint64_t b = (uint64_t)__double_as_longlong(x);
  const int e = (int)(b >> 52) & 0x7ff;
  const uint64_t mant = (b & ((1ull << 52) - 1)) | (1ull << 52);
  const int r = 1019 - e;
  uint64_t v;
  if (r <= 0) v = mant << ((-r) & 7);
  else v = r > 54 ? 0 : (mant + (1ull << (r - 1))) >> r;
  return (b >> 63) ? -(int64_t)v : (int64_t)v;
}

// The digits of two entries as fp16 pairs (x0 low, x1 high): out[s] for digit s.
__device__ __forceinline__ void dig_pair(double x0, double x1, uint32_t (&out)[DIG_N]) {
  // a bias of 128 in every digit's place (512 in the leading one's) makes the
  // digits plain bytes
  const uint64_t bias = 0x0200808080808080ull;
  const uint64_t w0 = (uint64_t)dig_fixed(x0) + bias, w1 = (uint64_t)dig_fixed(x1) + bias;
  const uint32_t l0 = (uint32_t)w0, l1 = (uint32_t)w1;
  const uint32_t h0 = (uint32_t)(w0 >> 32), h1 = (uint32_t)(w1 >> 32);
  const __half2 off = __half2half2(__ushort_as_half((unsigned short)0x6480));   // 1152
  // fp16 0x6400 + byte is 1024 + byte
  auto digit = [&](uint32_t pair) {
    const uint32_t u = (pair & 0x00ff00ffu) | 0x64006400u;
    __half2 h = *reinterpret_cast<const __half2 *>(&u);
    h = __hsub2(h, off);
    return *reinterpret_cast<const uint32_t *>(&h);
  };
  {
    const uint32_t u = (__byte_perm(h0, h1, 0x7632) & 0x03ff03ffu) | 0x64006400u;
    __half2 h = *reinterpret_cast<const __half2 *>(&u);
    h = __hsub2(h, __half2half2(__ushort_as_half((unsigned short)0x6600)));   // 1536
    out[0] = *reinterpret_cast<const uint32_t *>(&h);
  }
  out[1] = digit(__byte_perm(h0, h1, 0x0501));
  out[2] = digit(__byte_perm(h0, h1, 0x0400));
  out[3] = digit(__byte_perm(l0, l1, 0x0703));
  out[4] = digit(__byte_perm(l0, l1, 0x0602));
  out[5] = digit(__byte_perm(l0, l1, 0x0501));
  out[6] = digit(__byte_perm(l0, l1, 0x0400));
}

}  // namespace krr
