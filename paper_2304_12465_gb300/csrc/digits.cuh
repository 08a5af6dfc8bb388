// Float64 products of matrices, row by row, on the fp16 tensor cores by digits
// (an Ozaki-style splitting).
//
// Every row is scaled by the power of two 2^s that brings its norm into (1/2, 1],
// so that the errors below are relative to the norms of the two rows: many rows
// of a factor are small (points far from all pivots so far), and without their
// own scales the errors of a nearly sparse factor were two to eight times those
// of float64 sums.  A scaled entry is rounded once to the fixed-point integer v =
// round(2^56 x) and written as seven balanced base-256 digits, x = sum_s q_s
// 2^(-8 - 8 s), -128 <= q_s <= 127 (the leading one -512..511, for |x| below 2).
// Digits are exact in fp16; the product of digits s and t carries 2^(-16 - 8 (s +
// t)), so the pairs of one g = s + t share an accumulator.  Over n terms a pair of
// full digits stays within 2^14 n, a pair with one leading digit within 2^15
// sqrt(n) and the leading pair within 2^16 (the rows' norms, with room for the
// leading digits' rounding), so the sums of groups 3..6 (at most two pairs with a
// leading digit and five without) stay below 2^24 over DIG_LOW terms and those
// of groups 0..2 (one full pair) over DIG_HIGH, and the float32 accumulation is
// exact.  The 28 pairs with s + t <= 6 are kept; what is dropped is about
// 2^-59.6 sqrt(6 K) of the norms' product.  The accumulators go into one 64-bit
// total in units of 2^-60.
//
// A 128 x 64 x 16 product of float64 is 131072 multiply-adds: 69000 clocks of
// the float64 pipe of an SM (1.9 a clock), 1000 of its tensor cores as 28 digit
// products (4096 a clock).

#pragma once

#include <cuda_fp16.h>

#include "common.cuh"

namespace krr {

constexpr int DIG_N = 7;              // digits
constexpr int DIG_LOW = 160;          // terms between read-outs of groups 3..6
constexpr int DIG_HIGH = 640;         // and of groups 0..2
static_assert(5 * 16384.0 * DIG_LOW + 2 * 32768.0 * 12.65 <= 16777216.0, "groups 3..6");
static_assert(16384.0 * DIG_HIGH + 2 * 32768.0 * 25.3 + 65536.0 <= 16777216.0, "groups 0..2");

// The scale of a row from its squared norm: the largest s (at most DIG_MAX_SHIFT)
// with 2^s |row| <= 1 up to the rounding of the norm; 0 for zero and NaN.
constexpr int DIG_MAX_SHIFT = 400;
__device__ __forceinline__ int dig_shift(double n2) {
  if (!(n2 > 0.0) || !(n2 < 1e300)) return 0;
  // n2 (1 - 2^-20) lies below 2^(e - 1022)
  const int e = (int)(__double2hiint(n2 * (1.0 - 0x1p-20)) >> 20) & 0x7ff;
  return min((1022 - e) >> 1, DIG_MAX_SHIFT);
}

// round(2^(56 + s) x) + bias, top = 1023 - s, |2^s x| < 2 (0 + bias for |2^s x| <
// 2^-57): the mantissa as 2^5 times an integer, shifted right by the exponent's
// distance from 2 with one bit left, rounded there.
__device__ __forceinline__ uint64_t dig_fixed(double x, int top, uint64_t bias) {
  const uint64_t b = (uint64_t)__double_as_longlong(x);
  const int e = (int)(b >> 52) & 0x7ff;
  const uint64_t m5 = ((b & ((1ull << 52) - 1)) | (1ull << 52)) << 5;
  // (beyond 2, infinities and NaN: 0, without an undefined shift)
  const uint64_t v = ((m5 >> min((unsigned)(top - e), 63u)) + 1) >> 1;
  return (int64_t)b < 0 ? bias - v : bias + v;
}

// The digits of two entries of rows scaled by 2^s as fp16 pairs (x0 low, x1
// high): out[q] for digit q.  top = 1023 - s.
__device__ __forceinline__ void dig_pair(double x0, double x1, int top, uint32_t (&out)[DIG_N]) {
  // a bias of 128 in every digit's place (512 in the leading one's) makes the
  // digits plain bytes
  const uint64_t bias = 0x0200808080808080ull;
  const uint64_t w0 = dig_fixed(x0, top, bias), w1 = dig_fixed(x1, top, bias);
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
