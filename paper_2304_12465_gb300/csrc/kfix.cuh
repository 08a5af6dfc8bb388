// Float64-accurate kernel values in fixed-point arithmetic on the integer
// pipes.
//
// The float64 pipe of this GPU issues 1.9 DFMA a clock and SM (measured),
// the integer pipe 53 32 x 32 + 64-bit multiply-adds.  A float64 kernel entry
// costs 2d + 25 or so float64 operations (the differences, the squares and
// exp); the same entry in fixed point costs 5d + 60 integer instructions, and
// its intermediate sums are exact.
//
// A point set is centred and scaled by a factor that turns the exponent of
// the kernel into a plain sum, and rounded once to integers:
//   Gaussian  u = round(2^Q (x - ctr) sqrt(log2 e / 2) / sigma):  E = sum d^2 2^(-2Q)
//   Matern    u = round(2^Q (x - ctr) sqrt(5) / sigma):           q^2 = sum d^2 2^(-2Q)
//   Laplace   u = round(2^Q (x - ctr) log2 e / sigma):            E = sum |d| 2^(-Q)
// with d = u_i - u_j and kappa = 2^-E (Matern: the polynomial times exp(-q)).
// Gaussian and Matern coordinates have |u| < 2^57 and are kept as limbs
// u = 2^29 h + l, |l| <= 2^28, so that the three partial sums of squares
//   S1 = sum dh^2, S2 = sum dh dl, S3 = sum dl^2,  sum d^2 = 2^58 S1 + 2^30 S2 + S3
// of up to 32 coordinates are exact in 64 bits: five instructions (two
// subtractions, three multiply-adds) a coordinate.  Laplace coordinates have
// |u| < 2^60 as plain 64-bit integers; their differences are summed over groups
// of eight, whose two lowest bits are summed apart.
//
// Error: the coordinates are rounded once, to 2^-58 of the range's power of
// two (2^-61 for Laplace); everything after that is exact up to one
// rounding of E at 2^-55 and the mantissa of 2^-E, good to 2^-60, rounded to
// 53 bits.  Float64 arithmetic rounds every difference, square and sum and E
// itself at 2^-53 of E.  Point sets whose scaled half-range exceeds
// 2^kFixMaxExp (or that hold a non-finite value) keep the float64 kernels;
// the limits are where the coordinate rounding reaches the float64 one.
#pragma once

#include <cstdint>

#ifdef __CUDACC__
#define KRR_HD __host__ __device__ __forceinline__
#else
#include <cmath>
#include <cstring>
#define KRR_HD inline
#endif

namespace krr {

// Scaled half-range limit 2^e of each kernel function for the float64 products
// and for the float-float ones (about 2^-46 an entry), whose limits are where
// the coordinate rounding reaches that.
constexpr int kFixMaxExpGauss = 4, kFixMaxExpMatern = 6, kFixMaxExpLaplace = 5;
constexpr int kFixFFMaxExpGauss = 4, kFixFFMaxExpMatern = 5, kFixFFMaxExpLaplace = 9;
constexpr int kFixMinExp = 1;    // a smaller range gains nothing: E is kept at 2^-54
constexpr int kFixLimb = 29;
// Fraction bits of Laplace coordinates plus the range's exponent: |u| < 2^60, and
// eight differences below 2^61 stay within 64 bits.  From the second group on a
// sum keeps its two lowest bits apart (kFixL1Low): four shifted ones stay within
// 64 bits too.  With 58 bits and one plain sum, near pairs in 32 dimensions were
// off by up to 3.8 units of 2^-53 at the widest range, where the float64 formula
// is off by half a unit.  The float-float values, 8 units apart, keep 58 bits and
// one sum.
constexpr int kFixL1Bits = 60, kFixL1Group = 8, kFixL1Low = 2;
constexpr int kFixFFL1Bits = 58;
// The float-float products keep |u| < 2^53 with low limbs of 25 bits and leave
// out S3 but for its mean over low limbs: what is missing stays below d 2^(2 e
// - 56) of E (a fifth of 2^(2 e - 56) sqrt(d) in the mean square), and two
// multiply-adds a coordinate remain.  Pairs nearer than 2^-8 in E or q^2 take
// the whole sum (s1_near): there kappa is 1 but for a small difference, and
// equal points give exactly 1, as direct differences do.
constexpr int kFixFFLimb = 25;
constexpr int kFixNearExp = 8;
constexpr int kFixTab = 256;

// What the conversion and the products of one point set (or two: rows and
// columns) share.  Lives in device memory, so that no launch waits for the
// host; ok == 0 leaves the work to the float64 or float-float kernels.
struct FixScale {
  double ctr[32];
  double s_hi, s_lo;     // scale factor as an unevaluated sum
  double r2_scale;       // Matern: 2^(30 - 2 q)
  int64_t s1_max;        // Gaussian: see fix_exponent
  int64_t bias;          // float-float products: mean of S3 2^-26
  uint32_t s1_near;      // and the limit of S1 2^-32 below which S3 is formed
  int q;                 // fraction bits of u
  int r;                 // right shift to 54 fraction bits (Gaussian, Laplace)
  int limb;              // bits of the low limb (0: whole 64-bit integers)
  int ok;
};

// High word of a 64 x 64-bit product, low by at most 2: the product of the low
// halves is left out, which saves a multiply and its carries (the multiplies
// are what bounds the products).
KRR_HD uint64_t fix_mulhi(uint64_t a, uint64_t b) {
  const uint32_t al = (uint32_t)a, ah = (uint32_t)(a >> 32);
  const uint32_t bl = (uint32_t)b, bh = (uint32_t)(b >> 32);
  const uint64_t x = (uint64_t)al * bh, y = (uint64_t)ah * bl;
  return (uint64_t)ah * bh + (x >> 32) + (y >> 32);
}

// High word of a 32 x 32-bit product, by the wide multiply (the high-word one
// runs at half its rate).
KRR_HD uint32_t fix_mulhi32(uint32_t a, uint32_t b) {
#ifdef __CUDA_ARCH__
  uint64_t p;
  asm("mul.wide.u32 %0, %1, %2;" : "=l"(p) : "r"(a), "r"(b));
  return (uint32_t)(p >> 32);
#else
  return (uint32_t)(((uint64_t)a * b) >> 32);
#endif
}

KRR_HD double fix_bits_double(uint64_t b) {
#ifdef __CUDA_ARCH__
  return __longlong_as_double((long long)b);
#else
  double d;
  memcpy(&d, &b, 8);
  return d;
#endif
}

// round(2^(63 - j/256))
#ifdef __CUDACC__
__device__
#endif
static const uint64_t kFixExp2Tab[kFixTab] = {
    0x8000000000000000ull, 0x7fa765aca88f6453ull, 0x7f4f08ae3dc7c426ull, 0x7ef6e8da4b544f9aull,
    0x7e9f06067a4360baull, 0x7e47600890f223deull, 0x7deff6b672f84e24ull, 0x7d98c9e62113e1faull,
    0x7d41d96db915019dull, 0x7ceb252375c9cf9bull, 0x7c94acddaeea5d3aull, 0x7c3e7072d904a6ceull,
    0x7be86fb985689ddcull, 0x7b92aa886214411cull, 0x7b3d20b6399fc237ull, 0x7ae7d219f329b948ull,
    0x7a92be8a92436616ull, 0x7a3de5df36dcfeefull, 0x79e947ef1d320d2dull, 0x7994e4919db5d74eull,
    0x7940bb9e2cffd89dull, 0x78ecccec5bb84661ull, 0x78991853d684a285ull, 0x78459dac65f45bb5ull,
    0x77f25ccdee6d7ae6ull, 0x779f559070195e36ull, 0x774c87cc06d1812eull, 0x76f9f358ea0c5249ull,
    0x76a7980f6cca15c2ull, 0x765575c7fd81d5a0ull, 0x76038c5b260e5eeeull, 0x75b1dba18b9b4c20ull,
    0x75606373ee921c97ull, 0x750f23ab2a87593eull, 0x74be1c203627c62bull, 0x746d4cac2325a155ull,
    0x741cb5281e25ee34ull, 0x73cc556d6eadce5full, 0x737c2d55770fe711ull, 0x732c3cb9b459d38bull,
    0x72dc8373be41a454ull, 0x728d015d47136b40ull, 0x723db6501b9ed447ull, 0x71eea2262324cb0cull,
    0x719fc4b95f452d29ull, 0x71511de3ebec8913ull, 0x7102ad7fff41e9b4ull, 0x70b47367e994ae92ull,
    0x70666f76154a7089ull, 0x7018a18506ccf314ull, 0x6fcb096f5c782210ull, 0x6f7da70fce881bf9ull,
    0x6f307a412f074892ull, 0x6ee382de69bc7bf8ull, 0x6e96c0c284192610ull, 0x6e4a33c89d278e49ull,
    0x6dfddbcbed791babull, 0x6db1b8a7c714a92bull, 0x6d65ca379564e639ull, 0x6d1a1056dd26c382ull,
    0x6cce8ae13c57ebdbull, 0x6c8339b26a25494eull, 0x6c381ca636d99642ull, 0x6bed33988bcbfab5ull,
    0x6ba27e656b4eb57aull, 0x6b57fce8f09dd17full, 0x6b0daeff4fcde703ull, 0x6ac39484d5bae8c5ull,
    0x6a79ad55e7f6fd10ull, 0x6a2ff94f04b962b0ull, 0x69e6784cc2cd61bdull, 0x699d2a2bd181482aull,
    0x69540ec8f895722dull, 0x690b2601182b5e56ull, 0x68c26fb128b4cd63ull, 0x6879ebb63ae2edc6ull,
    0x683199ed779592caull, 0x67e97a341fca775bull, 0x67a18c678c8c8c61ull, 0x6759d0652ee352afull,
    0x6712460a8fc24072ull, 0x66caed354ff83222ull, 0x6683c5c3281ee6e9ull, 0x663ccf91e88a8873ull,
    0x65f60a7f79393e2eull, 0x65af7669d9c2cbe4ull, 0x6569132f21483ba7ull, 0x6522e0ad7e639312ull,
    0x64dcdec3371793d1ull, 0x64970d4ea8bf8766ull, 0x64516c2e47ff1623ull, 0x640bfb40a0b22959ull,
    0x63c6ba6455dcd8aeull, 0x6381a978219b628full, 0x633cc85ad5122fbdull, 0x62f816eb585de1edull,
    0x62b39508aa836d6full, 0x626f4291e1603dd5ull, 0x622b1f66299a6599ull, 0x61e72b64c690d8afull,
    0x61a3666d124bb204ull, 0x615fd05e7d6c83e4ull, 0x611c69188f1eb339ull, 0x60d9307ae507dd9aull,
    0x6096266533384a2bull, 0x60534ab7441b6546ull, 0x60109d50f86846d8ull, 0x5fce1e124712437cull,
    0x5f8bccdb3d398841ull, 0x5f49a98bfe1bc11cull, 0x5f07b404c304c9f1ull, 0x5ec5ec25db3f6a41ull,
    0x5e8451cfac061b5full, 0x5e42e4e2b073d935ull, 0x5e01a53f7974fd86ull, 0x5dc092c6adb825b8ull,
    0x5d7fad59099f22feull, 0x5d3ef4d75f2ff504ull, 0x5cfe69229605cef5ull, 0x5cbe0a1bab4226dfull,
    0x5c7dd7a3b17dcf75ull, 0x5c3dd19bd0ba1c1aull, 0x5bfdf7e546520f3eull, 0x5bbe4a6164eb92f4ull,
    0x5b7ec8f19468bbc9ull, 0x5b3f737751d915c8ull, 0x5b0049d42f6afbb6ull, 0x5ac14be9d45cf869ull,
    0x5a827999fcef3242ull, 0x5a43d2c67a54e0c0ull, 0x5a05575132a5cc20ull, 0x59c7071c20cfd70cull,
    0x5988e20954889245ull, 0x594ae7faf23eda52ull, 0x590d18d3330c7f1eull, 0x58cf747464a7f584ull,
    0x5891fac0e95612c8ull, 0x5854ab9b37dbd1e5ull, 0x581786e5db7022c2ull, 0x57da8c8373adc331ull,
    0x579dbc56b48521baull, 0x57611642662e4a33ull, 0x57249a29651adc07ull, 0x56e847eea1e80a49ull,
    0x56ac1f752150a563ull, 0x5670209ffc1f2e82ull, 0x56344b525f1ff495ull, 0x55f89f6f8b133af4ull,
    0x55bd1cdad49f699cull, 0x5581c377a44346f0ull, 0x5546932976483b15ull, 0x550b8bd3dab49cbdull,
    0x54d0ad5a753e077cull, 0x5495f7a0fd3bbb8eull, 0x545b6a8b3d990704ull, 0x542105fd14c7b869ull,
    0x53e6c9da74b29ab5ull, 0x53acb60762affaaeull, 0x5372ca67f774358full, 0x533906e05f045106ull,
    0x52ff6b54d8a89c75ull, 0x52c5f7a9b6df5b77ull, 0x528cabc35f4f799dull, 0x525387864abb4762ull,
    0x521a8ad704f3404full, 0x51e1b59a2cc8da3eull, 0x51a907b474015dc9ull, 0x5170810a9f48c7cfull,
    0x513821818624b40cull, 0x50ffe8fe12e750c4ull, 0x50c7d76542a25b72ull, 0x508fec9c251a267cull,
    0x50582887dcb8a7e1ull, 0x50208b0d9e8090dfull, 0x4fe91412b2006e83ull, 0x4fb1c37c7145d328ull,
    0x4f7a993048d088d7ull, 0x4f439513b785cc80ull, 0x4f0cb70c4ea39210ull, 0x4ed5feffb1b3d155ull,
    0x4e9f6cd3967fdba8ull, 0x4e69006dc503ba65ull, 0x4e32b9b417619617ull, 0x4dfc988c79d52661ull,
    0x4dc69cdceaa72a9cull, 0x4d90c68b7a20eb1eull, 0x4d5b157e4a7fc325ull, 0x4d25899b8fe8b365ull,
    0x4cf022c9905bfd32ull, 0x4cbae0eea3a8c63cull, 0x4c85c3f13360c4d5ull, 0x4c50cbb7bacbf4cbull,
    0x4c1bf828c6dc54b8ull, 0x4be7492af621abd6ull, 0x4bb2bea4f8bd5847ull, 0x4b7e587d905625d1ull,
    0x4b4a169b900c2d00ull, 0x4b15f8e5dc6cbab0ull, 0x4ae1ff436b663ff7ull, 0x4aae299b443c4a6bull,
    0x4a7a77d47f7b84b1ull, 0x4a46e9d646edbf6aull, 0x4a137f87d58e025bull, 0x49e038d0777ca5e0ull,
    0x49ad159789f37496ull, 0x497a15c47b39d53eull, 0x4947393eca98fcd6ull, 0x49147fee085028d6ull,
    0x48e1e9b9d588e19bull, 0x48af7689e44b44eaull, 0x487d2645f7725895ull, 0x484af8d5e2a06536ull,
    0x4818ee218a3358eeull, 0x47e70610e3393241ull, 0x47b5408bf36472e2ull, 0x47839d7ad1009a90ull,
    0x47521cc5a2e6a9e0ull, 0x4720be54a071ad01ull, 0x46ef821011734e6bull, 0x46be67e04e28717cull,
    0x468d6fadbf2dd4f3ull, 0x465c9960dd74bd4bull, 0x462be4e23237a6efull, 0x45fb521a56ef0042ull,
    0x45cae0f1f545eb73ull, 0x459a9151c70f0819ull, 0x456a632296394492ull, 0x453a564d3cc4b723ull,
    0x450a6abaa4b77ecdull, 0x44daa053c812abd2ull, 0x44aaf701b0c72feeull, 0x447b6ead78aad636ull,
    0x444c0740496d4294ull, 0x441cc0a35c8cf8eaull, 0x43ed9abffb4c6bc9ull, 0x43be957f7ea712b6ull,
    0x438fb0cb4f468808ull, 0x4360ec8ce577ae44ull, 0x433248adc91fdd02ull, 0x4303c51791b21550ull,
    0x42d561b3e6243d8aull, 0x42a71e6c7ce464afull, 0x4278fb2b1bce0d15ull, 0x424af7d9981f7e98ull,
    0x421d1461d66f2023ull, 0x41ef50adcaa0d899ull, 0x41c1aca777db771bull, 0x41942838f07e22a3ull,
    0x4166c34c5615d0ecull, 0x41397dcbd952c4a6ull, 0x410c57a1b9fe12f6ull, 0x40df50b846ef302bull,
    0x40b268f9de0183baull, 0x4085a050ec0a036aull, 0x4058f6a7ecccd5b6ull, 0x402c6be96af2fb58ull,
};

// u of one coordinate: 2^q (x - ctr)(s_hi + s_lo) rounded to an integer.  The
// difference and the product carry their rounding errors along (TwoSum,
// TwoProduct by fma), so u is within 1 of the exact value.
KRR_HD int64_t fix_coord(double x, double ctr, double s_hi, double s_lo,
                                             int q) {
  const double t = x - ctr;
  const double bb = t - x;
  const double te = (x - (t - bb)) + (-ctr - bb);
  const double p = t * s_hi;
  const double lo = fma(t, s_hi, -p) + fma(t, s_lo, te * s_hi);
  const double ps = ldexp(p, q), ls = ldexp(lo, q);
  const double pi = rint(ps);
  return (int64_t)pi + (int64_t)rint((ps - pi) + ls);
}

// u = 2^limb h + l with |l| <= 2^(limb - 1)
KRR_HD void fix_limbs(int64_t u, int limb, int32_t *h, int32_t *l) {
  const int64_t hh = (u + (1LL << (limb - 1))) >> limb;
  *h = (int32_t)hh;
  *l = (int32_t)(u - hh * (1LL << limb));
}

// The float-float products' E from 2^50 S1 + 2^26 A, A = S2 + S3 2^-26 or its
// mean.  A sum that falls below zero by the rounding of A is 0.
KRR_HD uint64_t fix_exponent_ff(int64_t S1, int64_t A, int r, int64_t s1_max) {
  const int64_t a = (A + (1LL << (r - 1))) >> r;
  const uint64_t b = (uint64_t)S1 << (24 - r);
  if (a < 0 && b < (uint64_t)-a) return 0;
  return S1 >= s1_max ? ~0ull : b + (uint64_t)a;
}

// E at 54 fraction bits from the partial sums of squares, rounded to nearest;
// all ones for E beyond 1022, where kappa leaves the float64 range (s1_max is
// that limit in units of S1: 1022 2^54 >> (28 - r)).
KRR_HD uint64_t fix_exponent(int64_t S1, int64_t S2, uint64_t S3, int r,
                                                 int64_t s1_max) {
  const int64_t A = S2 + (int64_t)(S3 >> 30);
  const uint64_t E = ((uint64_t)S1 << (28 - r)) + (uint64_t)((A + (1LL << (r - 1))) >> r);
  return S1 >= s1_max ? ~0ull : E;
}

// 2^-f at 2^-63, f the fraction of E (54 fraction bits).  The top 8 fraction bits select 2^(-j/256)
// from tab (units 2^-63); the rest, g < 2^-8, goes through 1 - 2^-g =
// g (c1 - g (c2 - g (c3 - g (c4 - g c5)))), c_i = ln(2)^i / i! (Taylor; the
// next term is below 2^-60): the inner coefficients in 32 bits, where their
// powers of g leave at most 2^-55 of the result to them, the outer two in 64.
KRR_HD uint64_t fix_exp2_mantissa(uint64_t E, const uint64_t *__restrict__ tab) {
  const int j = (int)(E >> 46) & 255;
  const uint64_t g = E & ((1ull << 46) - 1);               // units 2^-54
  const uint32_t gs = (uint32_t)(g >> 14);                  // units 2^-40
  // c4 - g c5 and c3 - g (c4 - g c5) at 2^-35
  const uint32_t t4 = 330476400u - (fix_mulhi32(gs, 45813757u) >> 8);
  const uint32_t t3 = 1907106652u - (fix_mulhi32(gs, t4) >> 8);
  // c2 - g t3 at 2^-62 (the product is at 2^-75)
  const uint64_t t2 = 0x0F5FDEFFC162C754ull - (((uint64_t)gs * t3) >> 13);
  const uint64_t G = g << 18;                               // units 2^-72
  // c1 - g t2 at 2^-63 (the high word of the product is at 2^-70)
  const uint64_t t1 = 0x58B90BFBE8E7BCD6ull - (fix_mulhi(G, t2) >> 7);
  const uint64_t p = fix_mulhi(G, t1);                      // 1 - 2^-g at 2^-71
  const uint64_t T = tab[j];
  return T - (fix_mulhi(T, p) >> 7);                        // 2^-f at 2^-63
}

// 2^-E as a float64 (0 below 2^-1021): bit 53 of the rounded mantissa carries
// into the exponent field.
KRR_HD double fix_exp2(uint64_t E, const uint64_t *__restrict__ tab) {
  const int n = (int)(E >> 54);
  const uint64_t m = fix_exp2_mantissa(E, tab);
  const uint64_t bits = ((uint64_t)(1021 - n) << 52) + ((m + 512) >> 10);
  return n > 1020 ? 0.0 : fix_bits_double(bits);
}

// E of the Laplace kernel at 54 fraction bits from the sum of |d| at
// 2^-(54 + r).
KRR_HD uint64_t fix_exponent_l1(uint64_t S, int r) {
  if (r < 0) return (S >> (64 + r)) ? ~0ull : S << -r;
  return r > 0 ? (S >> r) + ((S >> (r - 1)) & 1) : S;
}

// The same from the sums of the groups without their lowest bits (S, at
// 2^-(54 + r)) and of those bits (L, at 2^-(54 + kFixL1Low + r)).
KRR_HD uint64_t fix_exponent_l1_groups(uint64_t S, uint32_t L, int r) {
  S += L >> kFixL1Low;
  L &= (1u << kFixL1Low) - 1;
  if (r > 0) return fix_exponent_l1(S, r);
  if (r == 0) return S + (L >> 1);
  if (S >> (64 + r)) return ~0ull;
  return (S << -r) + (r == -1 ? (uint64_t)(L >> 1) : (uint64_t)L << (-r - kFixL1Low));
}

constexpr double kFixMaternEnd = 708.39;   // 1022 ln 2 = 708.396

// (1 + q + q^2/3) exp(-q) from the partial sums of squares; scale = 2^(30-2Q).
// The square root starts from the float32 reciprocal square root (2^-22) and
// takes one Goldschmidt step and a final residual correction in float64; q
// log2 e is a 64 x 64-bit fixed-point product.  E has ten integer bits, so it
// would wrap at q = 1024 ln 2 = 709.8, which opposite corners of the accepted
// range pass from d = 31 on (q up to 128 sqrt(d)): from E = 1022 on kappa, below
// 1e-302 there, is 0, as in the Gaussian and Laplace forms.
KRR_HD double fix_matern(int64_t S1, int64_t S2, uint64_t S3, double scale,
                                             const uint64_t *__restrict__ tab) {
  const int64_t A = S2 + (int64_t)(S3 >> 30);
  const double r2 = fma((double)S1, 268435456.0, (double)A) * scale;
  if (!(r2 > 1e-36)) return 1.0;
#ifdef __CUDA_ARCH__
  const double s0 = (double)rsqrtf((float)r2);
#else
  const double s0 = (double)(1.0f / sqrtf((float)r2));
#endif
  double g = r2 * s0, h = 0.5 * s0;
  const double e = fma(-g, h, 0.5);
  g = fma(g, e, g);
  h = fma(h, e, h);
  const double q = fma(fma(-g, g, r2), h, g);
  if (q >= kFixMaternEnd) return 0.0;
  uint64_t b;
#ifdef __CUDA_ARCH__
  b = (uint64_t)__double_as_longlong(q);
#else
  memcpy(&b, &q, 8);
#endif
  // q at 54 fraction bits: mantissa 2^52..2^53 at exponent field ex is worth
  // 2^(ex - 1075), so the shift to 2^-54 is ex - 1021
  const int sh = (int)(b >> 52) - 1021;
  const uint64_t mant = (b & ((1ull << 52) - 1)) | (1ull << 52);
  const uint64_t qf = sh >= 0 ? mant << sh : (mant + (1ull << (-sh - 1))) >> (-sh);
  const uint64_t L = 0xB8AA3B295C17F0BCull;                 // log2 e at 2^-63
#ifdef __CUDA_ARCH__
  const uint64_t hi = __umul64hi(qf, L);
#else
  const uint64_t hi = (uint64_t)(((unsigned __int128)qf * L) >> 64);
#endif
  const uint64_t E = (hi << 1) | ((qf * L) >> 63);
  return fma(q, fma(q, 1.0 / 3.0, 1.0), 1.0) * fix_exp2(E, tab);
}

}  // namespace krr
