// Fixed-point arithmetic of the FP64 operators on the integer pipe.
//
// This GPU issues 2 FP64 fused multiply-adds per clock and SM (measured: 1.99)
// but about 25 32x32->64-bit integer multiply-adds (mad.wide, measured with varying
// operands).  A complex product u b with 62-bit fixed-point values costs 12 of those
// and 9 integer additions, against 4 FP64 multiply-adds: per bond of a checkerboard
// factor 1.2 clocks against 4.2 (measured, 363 threads, 12 sites per thread).
//
// Representation.  A slice is scaled by one power of two: with E the smallest
// integer such that every component is below 2^E, the value x is held as the 64-bit
// integer round(x 2^(F - E)), where F leaves room for the growth of a component through
// the operator (fx_fraction_bits in fx_strip.cuh).  For M^dagger M at dtau t = 0.1, F =
// 59: one unit is 2^-59 of the power of two above the slice's largest component (FP64
// rounds each operation at 2^-53 of its own result), and the rounding of a complex
// product is about 0.3 units.  Errors (2-norm) of Gaussian vectors against quad precision:
// M^dagger M 4.9e-17 (FP64 kernel 1.5 to 2.0e-16), M 6.0e-17 (1.4e-16).  They are the same for
// every element of a slice, where FP64's follow the element's size: see fx_uneven.
//
// A factor u of modulus below 1/2 is held as round(u 2^64) in two signed 32-bit limbs,
// u 2^64 = h 2^32 + l with -2^31 < l < 2^31 (so the neglected product of two low
// limbs, below 1/4 unit, has no bias, and -u is formed limb by limb).  b is split the same way (its low limb is its
// low word), hence u b = (uh bh) + ((uh bl + ul bh) >> 32): the cross terms add up in
// one 64-bit accumulator that starts at 2^31 (rounding) and gives its high word.
// That accumulator stays below 2^63 for the F of fx_fraction_bits.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>
#include <cstring>

namespace hqmc {

constexpr int kFxZero = -4096;      // exponent of an all-zero slice
constexpr int kFxBad = 1 << 20;     // exponent of a slice with an infinity or a NaN
constexpr int kFxBadLink = INT32_MIN;  // high limb of a link whose angle is not finite

// The arithmetic below is plain integer code for host and device (the CPU tests
// compile it for the host).
#define HQMC_HD __host__ __device__ __forceinline__

HQMC_HD long long fx_madw(int a, int b, long long c) {
#if defined(__CUDA_ARCH__)
  long long d;
  asm("mad.wide.s32 %0, %1, %2, %3;" : "=l"(d) : "r"(a), "r"(b), "l"(c));
  return d;
#else
  return (long long)a * b + c;
#endif
}
HQMC_HD long long fx_bits(double x) {
#if defined(__CUDA_ARCH__)
  return __double_as_longlong(x);
#else
  long long b;
  memcpy(&b, &x, 8);
  return b;
#endif
}
HQMC_HD double fx_from_bits(long long b) {
#if defined(__CUDA_ARCH__)
  return __longlong_as_double(b);
#else
  double x;
  memcpy(&x, &b, 8);
  return x;
#endif
}
HQMC_HD int fx_clz(long long a) {
#if defined(__CUDA_ARCH__)
  return __clzll(a);
#else
  return __builtin_clzll((unsigned long long)a);
#endif
}
HQMC_HD unsigned long long fx_umulhi(unsigned long long a, unsigned long long b) {
#if defined(__CUDA_ARCH__)
  return __umul64hi(a, b);
#else
  return (unsigned long long)(((unsigned __int128)a * b) >> 64);
#endif
}
// Balanced limbs of v: v = fx_hi(v) 2^32 + fx_lo(v), the low limb signed.
HQMC_HD int fx_lo(long long v) { return (int)v; }
HQMC_HD int fx_hi(long long v) {
  return (int)(v >> 32) + (int)((uint32_t)v >> 31);
}
constexpr long long kFxRound = 1ll << 31;

// a + s b (real s in limbs)
HQMC_HD long long fx_fma(long long a, int sh, int sl, long long b) {
  const int bh = fx_hi(b), bl = fx_lo(b);
  const long long h = fx_madw(sh, bh, a);
  const long long c = fx_madw(sl, bh, fx_madw(sh, bl, kFxRound));
  return h + (long long)(int)(c >> 32);
}

// a + u b
HQMC_HD longlong2 cfma(longlong2 a, int4 u, longlong2 b) {  // u = (re h, re l, im h, im l)
  const int ch = fx_hi(b.x), cl = fx_lo(b.x), dh = fx_hi(b.y), dl = fx_lo(b.y);
  const int nh = -u.z, nl = -u.w;
  long long h = fx_madw(nh, dh, fx_madw(u.x, ch, a.x));
  long long c = fx_madw(nl, dh, fx_madw(nh, dl, fx_madw(u.y, ch, fx_madw(u.x, cl, kFxRound))));
  const long long re = h + (long long)(int)(c >> 32);
  h = fx_madw(u.z, ch, fx_madw(u.x, dh, a.y));
  c = fx_madw(u.w, ch, fx_madw(u.z, cl, fx_madw(u.y, dh, fx_madw(u.x, dl, kFxRound))));
  return make_longlong2(re, h + (long long)(int)(c >> 32));
}
// a + conj(u) b
HQMC_HD longlong2 cfmac(longlong2 a, int4 u, longlong2 b) {
  return cfma(a, make_int4(u.x, u.y, -u.z, -u.w), b);
}

// ---------------------------------------------------------------------------
// Conversions (integer only: the FP64 pipe converts at the rate of its other work).

// Key of a double for the slice maximum: monotone in |x|, 0 only for zero.
HQMC_HD uint32_t fx_key(double x) {
  const long long b = fx_bits(x);
  return ((uint32_t)(b >> 32) & 0x7fffffffu) | ((uint32_t)b != 0 ? 1u : 0u);
}
// Exponent of a slice from its largest key.
HQMC_HD int fx_exponent(uint32_t key) {
  const int ex = (int)(key >> 20);
  return key == 0 ? kFxZero : ex == 2047 ? kFxBad : (ex == 0 ? 1 : ex) - 1022;
}

// Whether a slice falls off too far to be held at one scale: a strip of it has its largest
// component (strip: its key) below 2^-6 of the slice's (key).  A unit is 2^-58 of the slice's largest component or
// less and a result is off by a few units (5e-17 of a dense vector's 2-norm), FP64
// arithmetic by about 2e-16 of the values nearby: at 2^-6 the two meet.  Such slices
// (point sources, sparse or localised vectors) are computed in FP64 where a caller sees
// the result itself.  Gaussian vectors, M^dagger of them and solutions on ordered and
// on random fields (18^2 x 180 ... 66^2 x 660) stay above 2^-5.6.
HQMC_HD bool fx_uneven(uint32_t strip, uint32_t key, unsigned bits = 6) { return strip + (bits << 20) < key; }

// Shift base of a slice of exponent E (an all-zero slice converts like the smallest one).
HQMC_HD int fx_shift_base(int E, int F) { return 1085 - F + (E < -1021 ? -1021 : E); }

// round(x 2^(F - E)) for |x| < 2^E; s0 = fx_shift_base(E, F).
HQMC_HD long long fx_from_double(double x, int s0) {
  const long long bits = fx_bits(x);
  const int hi = (int)(bits >> 32);
  int ex = (hi >> 20) & 0x7ff;
  unsigned long long a = ((unsigned long long)bits << 10) & 0x3fffffffffffffffull;  // 52 bits of it
  if (ex) a |= 1ull << 62;
  else ex = 1;  // a denormal (or zero)
  const int s = s0 - ex;  // >= 63 - F >= 1
  const unsigned long long r = s > 63 ? 0ull : ((a >> (s - 1)) + 1) >> 1;
  const long long sg = (long long)(hi >> 31);
  return ((long long)r ^ sg) - sg;
}

// v 2^e rounded to the nearest double (ties to even); the result's exponent must be normal.
HQMC_HD double fx_to_double_normal(long long v, int e) {
  const long long sg = v >> 63;
  const unsigned long long a = (unsigned long long)((v ^ sg) - sg);
  if (a == 0) return 0.0;
  const int lz = fx_clz((long long)a);              // >= 1
  const unsigned long long b = a << (lz - 1);       // in [2^62, 2^63)
  unsigned long long m = (b + 512) >> 10;
  if (((unsigned)b & 1023u) == 512u) m &= ~1ull;    // a tie
  const unsigned long long bits = ((unsigned long long)(1085 - lz + e) << 52) + m;
  return fx_from_bits((long long)(bits | ((unsigned long long)sg & (1ull << 63))));
}
// The same for any e (uniform over a block): far from the middle of the exponent range the
// result is formed 2^512 away and scaled, so that it underflows and overflows as FP64
// does.  The exponent of a product of two slices goes far beyond what one such step
// covers (to -2160 and 2000); below 2^-1300 every v is zero, above 2^1100 infinite.
HQMC_HD double fx_to_double(long long v, int e) {
  if (e > -800 && e < 800) return fx_to_double_normal(v, e);
  return e < 0 ? fx_to_double_normal(v, (e < -1300 ? -1300 : e) + 512) * 0x1p-512
               : fx_to_double_normal(v, (e > 1100 ? 1100 : e) - 512) * 0x1p512;
}

// v 2^-n rounded, n >= 0 (uniform over a block).
HQMC_HD long long fx_shr(long long v, int n) {
  if (n == 0) return v;
  if (n > 62) return 0;
  return (v + (1ll << (n - 1))) >> n;
}

// Place of the link of site (x, y) in direction c in a slice's table: each family and
// parity in a plane of its own, so that a warp, whose threads own neighbouring column
// pairs, reads 512 contiguous bytes.  (Two links side by side per site, as in the FP64
// table, made every read fetch twice what it used.)
//   x-bonds: [x & 1][y][x / 2]; y-bonds, after them: [y & 1][y / 2][x & 1][x / 2].
HQMC_HD int fx_link_index(int L, int x, int y, int c) {
  const int Lh = L >> 1;
  if (c == 0) return ((x & 1) * L + y) * Lh + (x >> 1);
  return 2 * L * Lh + (((y & 1) * Lh + (y >> 1)) * 2 + (x & 1)) * Lh + (x >> 1);
}

// Limbs of the link (re, im), in units of 2^-64.  conj(u) and -u are formed limb by limb,
// and a low limb of -2^31 has no negative in 32 bits: such a component moves by one unit
// (left as it is, one link in 2^31 had cross terms of the wrong sign, 2^-32 of the product).
HQMC_HD int4 fx_link_limbs(long long re, long long im) {
  re += fx_lo(re) == INT32_MIN ? 1 : 0;
  im += fx_lo(im) == INT32_MIN ? 1 : 0;
  return make_int4(fx_hi(re), fx_lo(re), fx_hi(im), fx_lo(im));
}

// By integers: the slices that take FP64 need the FP64 pipe for their products.
HQMC_HD double2 fx_link_to_double(int4 u) {
  if (u.x == kFxBadLink) {
    const double nan = fx_from_bits(0x7ff8000000000000ll);
    return make_double2(nan, nan);
  }
  return make_double2(fx_to_double_normal(((long long)u.x << 32) + u.y, -64),
                      fx_to_double_normal(((long long)u.z << 32) + u.w, -64));
}

// ---------------------------------------------------------------------------
// Angles.  theta / 2 pi is formed in fixed point from the 53-bit significand and a
// 96-bit 1 / 2 pi, exact to 2^-64 of a turn for |theta| < 2^28; then sine and cosine by
// the addition theorem: the nearest of 256 table angles, and the Taylor series of the
// rest (|d| <= pi / 256, omitted terms below 2^-66).  Absolute error below 2^-60.
static const longlong2 kFxEighth[33] = {  // round(2^62 (cos, sin)(2 pi k / 256)), k <= 32 (an eighth of a turn)
    {0x4000000000000000ll, 0x0000000000000000ll},
    {0x3ffb10c1099a1976ll, 0x0192155f7a3667e0ll},
    {0x3fec43c6f2dafbc7ll, 0x0323ecbe21bb027dll},
    {0x3fd39b5a0310742all, 0x04b54824b3867d73ll},
    {0x3fb11b47a24a4b3cll, 0x0645e9af0a6d0af8ll},
    {0x3f84c8e1c33fa68fll, 0x07d59395aa5cc38dll},
    {0x3f4eaafe114a2d43ll, 0x0964083747309d11ll},
    {0x3f0ec9f4e297526bll, 0x0af10a22459fe32all},
    {0x3ec52f9feeb96056ll, 0x0c7c5c1e34d3055bll},
    {0x3e71e758c9cb118all, 0x0e05c1353f27b17ell},
    {0x3e14fdf72461ae55ll, 0x0f8cfcbd90af8d58ll},
    {0x3dae81ced092c67all, 0x1111d262b1f67761ll},
    {0x3d3e82ad8c5bb4bbll, 0x1294062ed59f05a9ll},
    {0x3cc511d891c223ddll, 0x14135c9417660143ll},
    {0x3c424209ed0dc97fll, 0x158f9a75ab1fdcfell},
    {0x3bb6276d998478c2ll, 0x17088530fa459eafll},
    {0x3b20d79e651a8c51ll, 0x187de2a6aea962d2ll},
    {0x3a8269a29b927359ll, 0x19ef7943a8ed8a2ell},
    {0x39daf5e8798ee5e2ll, 0x1b5d1009e15cc02bll},
    {0x392a96426823e9edll, 0x1cc66e9931c45e17ll},
    {0x387165e3017b61a4ll, 0x1e2b5d3806f63b1ell},
    {0x37af8158df2a533fll, 0x1f8ba4dbf89ab9fbll},
    {0x36e5068a32dc7b22ll, 0x20e70f3245ffdb2dll},
    {0x361214b02a03ff37ll, 0x223d66a836964508ll},
    {0x3536cc521d434606ll, 0x238e76735cd190d9ll},
    {0x34534f408c4f03bbll, 0x24da0a99ba25bd51ll},
    {0x3367c08fe70e8168ll, 0x261feff9c2e069c2ll},
    {0x3274449324c7f69fll, 0x275ff45240a17279ll},
    {0x317900d62a2e816all, 0x2899e64a123bac30ll},
    {0x30761c17ff2edba4ll, 0x29cd9577c7cbd228ll},
    {0x2f6bbe44d55f5dbcll, 0x2afad26919d93f45ll},
    {0x2e5a106fdfff2c87ll, 0x2c216eaa3a59bdb7ll},
    {0x2d413cccfe779921ll, 0x2d413cccfe779921ll},
};

// Ranges of |theta| by the high word of the double (a comparison on the FP64 pipe would
// cost as much as the rest of a wrap to float).
HQMC_HD uint32_t fx_abs_hi(double theta) { return (uint32_t)(fx_bits(theta) >> 32) & 0x7fffffffu; }
constexpr uint32_t kFxBelowPi = 0x400921fbu;     // below: |theta| < 3.14159202
constexpr uint32_t kFxMaxAngle = 0x41b00000u;    // 2^28; from here the caller uses the library's functions
constexpr uint32_t kFxNotFinite = 0x7ff00000u;

// theta / 2 pi mod 1, as a signed 64-bit fraction of a turn; |theta| < 2^28.
HQMC_HD long long fx_turns(double theta) {
  constexpr unsigned long long kHi = 0xa2f9836e4e441529ull;  // 2^98 / 2 pi, the high 64 of 96 bits
  constexpr unsigned kLo = 0xfc2757d1u;                      // and its low 32
  const long long bits = fx_bits(theta);
  int ex = (int)((bits >> 52) & 0x7ff);
  unsigned long long m = (unsigned long long)bits & 0xfffffffffffffull;
  if (ex) m |= 1ull << 52;
  else ex = 1;
  // P = m (kHi 2^32 + kLo) = theta / 2 pi 2^(98 + 1075 - ex); the fraction wants P >> s
  const unsigned long long b0 = (m & 0xffffffffull) * kLo, b1 = (m >> 32) * kLo;
  const unsigned long long low = b1 + (b0 >> 32);      // (m kLo) >> 32
  unsigned long long p0 = m * kHi, p1 = fx_umulhi(m, kHi);  // (p1, p0) + low = P >> 32
  const unsigned long long q0 = p0 + low;
  p1 += q0 < p0 ? 1ull : 0ull;
  const int s = 1077 - ex;  // of P >> 32; ex <= 1023 + 27, so s >= 27
  unsigned long long f;
  if (s < 64) f = (q0 >> s) | (p1 << (64 - s));
  else if (s < 128) f = s == 64 ? p1 : p1 >> (s - 64);
  else f = 0;
  return bits < 0 ? -(long long)f : (long long)f;
}

// The table angle k of a full turn in 256 parts, scaled by 2^62.
__host__ __device__ inline longlong2 fx_table_angle(int k, const longlong2* eighth) {
  const int j = k & 63;
  longlong2 e = eighth[j <= 32 ? j : 64 - j];
  if (j > 32) e = make_longlong2(e.y, e.x);
  switch ((k >> 6) & 3) {
    case 1: return make_longlong2(-e.y, e.x);
    case 2: return make_longlong2(-e.x, -e.y);
    case 3: return make_longlong2(e.y, -e.x);
    default: return e;
  }
}

// floor(a b / 2^64), signed
HQMC_HD long long fx_mulhi(long long a, long long b) {
#if defined(__CUDA_ARCH__)
  return __mul64hi(a, b);
#else
  return (long long)(((__int128)a * b) >> 64);
#endif
}
HQMC_HD int fx_mulhi32(int a, int b) {
#if defined(__CUDA_ARCH__)
  return __mulhi(a, b);
#else
  return (int)(((long long)a * b) >> 32);
#endif
}
HQMC_HD unsigned fx_umulhi32(unsigned a, unsigned b) {
  return (unsigned)(((unsigned long long)a * b) >> 32);
}

// (d.x u.y - d.y u.x) 2^(shift - 64), rounded.  d.y is negated before it is split: its low
// limb may be -2^31, which has no negative.
HQMC_HD long long fx_im(longlong2 d, longlong2 u, int shift) {
  const long long ny = -d.y;
  const int dxh = fx_hi(d.x), dxl = fx_lo(d.x), dyh = fx_hi(ny), dyl = fx_lo(ny);
  const int uxh = fx_hi(u.x), uxl = fx_lo(u.x), uyh = fx_hi(u.y), uyl = fx_lo(u.y);
  const long long hh = fx_madw(dyh, uxh, fx_madw(dxh, uyh, 0));
  // the cross terms and the high words of the low limbs' products, with half a unit of the result
  const long long low = (long long)fx_mulhi32(dxl, uyl) + fx_mulhi32(dyl, uxl) + (1ll << (31 - shift));
  const long long c = fx_madw(dyl, uxh, fx_madw(dyh, uxl, fx_madw(dxl, uyh, fx_madw(dxh, uyl, low))));
  return (hh << shift) + (c >> (32 - shift));
}

// s (cos, sin) of f turns for a table of s (cos, sin)(2 pi k / 256), in the table's units.
HQMC_HD longlong2 fx_cossin(long long f, const longlong2* __restrict__ table) {
  // nearest table angle k, rest r in [-2^55, 2^55) (units of 2^-64 turn)
  const unsigned long long fr = (unsigned long long)f + (1ull << 55);
  const longlong2 t = table[(int)(fr >> 56)];
  const long long r = (long long)(fr & ((1ull << 56) - 1)) - (1ll << 55);
  // d = 2 pi r 2^-64 <= pi / 256, in units of 2^-68: 32 pi r = 101 r - (101 - 32 pi) r
  const long long d = 101 * r - fx_mulhi(r, 0x7812aeef4b9ee59ell);
  const long long u = fx_mulhi(d, d);        // d^2 in units of 2^-72
  const unsigned v = (unsigned)(u >> 28);    // d^2 in units of 2^-44 (below 2^31.4)
  // sin d = d (1 - u ws), cos d = 1 - u wc with, in units of 2^-63,
  // ws = 1/6 - u (1/120 - u/5040), wc = 1/2 - u (1/24 - u/720); the brackets in 32 bits
  // (units of 2^-38 and 2^-36): their terms are 2^-17 and less of ws and wc
  const unsigned bs = 2290649225u - fx_umulhi32(v, 13315u);
  const unsigned bc = 2863311531u - fx_umulhi32(v, 23302u);
  const long long ws = 0x1555555555555555ll - (long long)(((unsigned long long)v * bs) >> 19);
  const long long wc = (1ll << 62) - (long long)(((unsigned long long)v * bc) >> 17);
  const long long us = fx_mulhi(u, ws), uc = fx_mulhi(u, wc);  // units of 2^-71
  const long long sd = d - (fx_mulhi(d, us) >> 7);             // sin d in units of 2^-68
  // products with the table in units of 2^-4 of its own
  const long long c = (fx_mulhi(t.x, uc) >> 3) + fx_mulhi(t.y, sd);
  const long long s = (fx_mulhi(t.y, uc) >> 3) - fx_mulhi(t.x, sd);
  return make_longlong2(t.x - ((c + 8) >> 4), t.y - ((s + 8) >> 4));
}

// sin d and 1 - cos d in FP64 from a table of 2^62 (cos, sin)(2 pi k / 256).  Fixed point
// is exact to 2^-60; below 2^-7, where that would cost relative precision, the series in
// FP64 (the omitted terms are below 2^-54 of the result).
__device__ __forceinline__ double fx_sin(double d, const longlong2* __restrict__ table) {
  const uint32_t a = fx_abs_hi(d);
  if (a < 0x3f800000u) {
    const double s = d * d;
    return fma(s * d, fma(s, fma(s, -1.0 / 5040.0, 1.0 / 120.0), -1.0 / 6.0), d);
  }
  if (a < kFxMaxAngle) return fx_to_double_normal(fx_cossin(fx_turns(d), table).y, -62);
  return sin(d);
}
__device__ __forceinline__ double fx_versine(double d, const longlong2* __restrict__ table) {
  const uint32_t a = fx_abs_hi(d);
  if (a < 0x3f800000u) {
    const double s = d * d;
    return s * fma(s, fma(s, fma(s, -1.0 / 40320.0, 1.0 / 720.0), -1.0 / 24.0), 0.5);
  }
  if (a < kFxMaxAngle) return fx_to_double_normal((1ll << 62) - fx_cossin(fx_turns(d), table).x, -62);
  return 1.0 - cos(d);
}

// theta wrapped to [-pi, pi] and rounded to float (the angle the FP32 kernels take).
__device__ __forceinline__ float fx_wrap_float(double theta) {
  const uint32_t a = fx_abs_hi(theta);
  if (a < kFxBelowPi) {
    const long long bits = fx_bits(theta);
    const unsigned ex = (unsigned)(bits >> 52) & 0x7ffu;
    if (ex <= 897u) return (float)theta;  // denormal as a float, or zero
    const unsigned long long m = (unsigned long long)bits & 0x7fffffffffffffffull;
    // round to nearest even at bit 29; the carry moves into the exponent
    const unsigned q = (unsigned)((m + 0xfffffffull + ((m >> 29) & 1ull)) >> 29) - (896u << 23);
    return __uint_as_float(q | ((unsigned)(bits >> 32) & 0x80000000u));
  }
  if (a < kFxMaxAngle) {
    const long long f = fx_turns(theta);
    return __ll2float_rn(f - fx_mulhi(f, 0x36f0255dde973dcbll)) * 0x1p-61f;  // f pi / 4
  }
  const double w = 6.283185307179586, iw = 0.15915494309189535;
  return (float)(theta - w * rint(theta * iw));
}

}  // namespace hqmc
