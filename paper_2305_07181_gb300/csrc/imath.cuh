// Logarithm and exponential of the nodal states in integer arithmetic.
//
// On GB300 one float64 instruction of a warp occupies its scheduler's float64
// pipe for ~76 clocks, an integer or float32 one for 1 to 2.  The table-driven
// float64 log and exp (fmath.cuh) take 17 and 14 float64 instructions; these
// take none, ~60 integer and float32 instructions each, which hide behind the
// float64 work around them.  Numbers are fixed point, 64-bit integers of
// 2^-57: absolute error of the logarithm below 2^-57.3 whatever its size (half
// a unit, and 10 units of 2^-62 from the terms below), so a power formed from
// it (q = rho^a p^b) is good to a few 2^-56 relative, while a float64 logarithm
// of size 2 alone carries 2^-53 into the exponential.
//
//   log:  x = 2^k m, m in [1, 2); j the top 8 bits of m's fraction;
//         z = m r_j / 2^14 - 1 exactly (14-bit r_j ~ 2^14/m: the 67-bit
//         product modulo 2^64), |z| < 2^-8.9;
//         ln x = k ln 2 + T_j + z - z^2 (1/2 - z/3) - z^4 (1/4 - z/5 + z^2/6),
//         T_j = -ln(r_j / 2^14) tabulated; the last term, below 2^-37, in
//         float32 (error below 6 units of 2^-62).  The terms are added in units
//         of 2^-62 and rounded once; log_fixed62, near 1, keeps those units.
//   exp:  X = N ln2/512 + r, |r| < 2^-10.5, N = 512 K + j;
//         exp X = 2^K 2^(j/512) (1 + r + r^2/2 + r^3/6 (1 + r/4 + r^2/20)),
//         the cubic term, below 2^-34, in float32.
// Method: table lookup and short series as in Tang (ACM TOMS 1989, 1990), in
// fixed point; tables (6.5 KB) by gen_imath_tables.py.
// Domain: log of normal x in [2^-90, 2^90), exp of |X| < 64; the callers take
// the float64 functions outside it.
#pragma once

#include <stdint.h>

#ifdef __CUDACC__
#define IM_FN __device__ __forceinline__
#define IM_TABLE __device__ const
#define IM_LOAD(p) __ldg(p)
#else  // host build of the same arithmetic (tests)
#include <cmath>
#include <cstring>
#define IM_FN static inline
#define IM_TABLE static const
#define IM_LOAD(p) (*(p))
static inline long long __mul64hi(long long a, long long b) { return (long long)(((__int128)a * b) >> 64); }
static inline unsigned long long __umul64hi(unsigned long long a, unsigned long long b) {
  return (unsigned long long)(((unsigned __int128)a * b) >> 64);
}
static inline int __clzll(long long x) { return x ? __builtin_clzll((unsigned long long)x) : 64; }
static inline int __float2int_rn(float x) { return (int)std::lrintf(x); }
static inline float __int2float_rn(int x) { return (float)x; }
static inline long long __double_as_longlong(double x) {
  long long b;
  std::memcpy(&b, &x, 8);
  return b;
}
static inline double __longlong_as_double(long long b) {
  double x;
  std::memcpy(&x, &b, 8);
  return x;
}
#endif

#include "imath_tables.h"

namespace esplit {
namespace im {

constexpr int UNIT = 57;  // fixed point: multiples of 2^-57

// a b / 2^60 (a fixed point, b of unit 2^-60); false when its size is not below 32
IM_FN bool mul_q60(long long a, long long b, long long& out) {
  const long long hi = __mul64hi(a, b);
  out = (long long)(((unsigned long long)hi << 4) | (((unsigned long long)a * (unsigned long long)b) >> 60));
  return (unsigned long long)(hi + (1LL << 58)) < (1ULL << 59);
}

// ln x in units of 2^-57; false (and nothing written) outside [2^-90, 2^90)
IM_FN bool log_fixed(double x, long long& L) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  const int k = (int)(b >> 52) - 1023;  // negative x: k >= 1025
  if ((unsigned)(k + 90) >= 180u) return false;
  const int j = (int)(b >> 44) & 255;
  const unsigned long long M = (b & 0xFFFFFFFFFFFFFULL) | 0x10000000000000ULL;
  const long long z = (long long)(M * (unsigned long long)IM_LOAD(&LOG_R[j]));  // unit 2^-66 (2^66 = 0 mod 2^64)
  const long long a = (long long)((unsigned long long)z << 5);                  // unit 2^-71, |a| < 2^62.2
  const long long h = __mul64hi(a, a);                                          // z^2, unit 2^-78
  const long long w = (1LL << 61) - __mul64hi(a, 0x2AAAAAAAAAAAABLL);           // 1/2 - z/3, unit 2^-62 (2^55 / 3)
  const long long s = __mul64hi(h, w);                                          // z^2 (1/2 - z/3), unit 2^-76
  const float zf = __int2float_rn((int)(a >> 32)) * 0x1p-39f, z2 = zf * zf;
  const int t = __float2int_rn(z2 * z2 * (0.25f + zf * (zf * 0.16666667f - 0.2f)) * 0x1p+62f);
  const long long low = (((long long)k * LN2_LO) >> 27) + IM_LOAD(&LOG_T[j]) + (z >> 4) - (s >> 14) - t;  // unit 2^-62
  L = (long long)k * LN2_HI + ((low + 16) >> 5);
  return true;
}

// ln x in units of 2^-62 for x in [1/4, 4): absolute error below 2^-59
IM_FN bool log_fixed62(double x, long long& L) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  const int k = (int)(b >> 52) - 1023;
  if ((unsigned)(k + 2) >= 4u) return false;
  const int j = (int)(b >> 44) & 255;
  const unsigned long long M = (b & 0xFFFFFFFFFFFFFULL) | 0x10000000000000ULL;
  const long long z = (long long)(M * (unsigned long long)IM_LOAD(&LOG_R[j]));
  const long long a = (long long)((unsigned long long)z << 5);
  const long long h = __mul64hi(a, a);
  const long long w = (1LL << 61) - __mul64hi(a, 0x2AAAAAAAAAAAABLL);
  const long long s = __mul64hi(h, w);
  const float zf = __int2float_rn((int)(a >> 32)) * 0x1p-39f, z2 = zf * zf;
  const int t = __float2int_rn(z2 * z2 * (0.25f + zf * (zf * 0.16666667f - 0.2f)) * 0x1p+62f);
  L = (long long)k * LN2_62 + IM_LOAD(&LOG_T[j]) + ((z + 8) >> 4) - ((s + (1LL << 13)) >> 14) - t;
  return true;
}

// exp(X 2^-57), any X (the value below 64)
IM_FN double exp_fixed(long long X) {
  // N = X 512/ln 2 rounded, from the upper word (unit 2^-25)
  const long long Nw = (long long)(int)(X >> 32) * INV_LN2_512 + (1LL << 44);
  const int N = (int)(Nw >> 45);
  const long long r = X - (long long)N * LN2_512_HI - (((long long)N * LN2_512_LO) >> 32);
  const long long a = (long long)((unsigned long long)r << 15);  // unit 2^-72, |a| < 2^61.6
  const long long h = __mul64hi(a, a);                           // r^2, unit 2^-80
  const float rf = __int2float_rn((int)(a >> 32)) * 0x1p-40f;
  const float c = rf * rf * rf * (0.16666667f + rf * (0.041666668f + rf * 0.008333334f));
  // exp(r) - 1, unit 2^-63
  const long long e = (long long)((unsigned long long)r << 6) + (h >> 18) + __float2int_rn(c * 0x1p+63f);
  const unsigned long long T = IM_LOAD(&EXP_T[N & 511]);  // unit 2^-62
  // T e, e signed
  const long long p = (long long)(__umul64hi(T, (unsigned long long)e) - (e < 0 ? T : 0ULL));
  const unsigned long long R = T + ((unsigned long long)p << 1);
  const int lz = __clzll((long long)R);  // 0, 1 or 2
  const unsigned long long n = R << lz;
  const unsigned long long m = (n >> 11) + ((n >> 10) & 1ULL);
  return __longlong_as_double((long long)(m + ((unsigned long long)(1023 + (N >> 9) - lz) << 52)));
}

// |x| < 2^-4 in units of 2^-66, truncated
IM_FN long long small_to_fixed(double x) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  const int sh = 1018 - ((int)(b >> 52) & 0x7ff);  // x = M 2^(-57 - sh), M < 2^53
  const unsigned long long M = (b & 0xFFFFFFFFFFFFFULL) | 0x10000000000000ULL;
  const unsigned long long v = sh > 62 ? 0ULL : ((M << 9) >> sh);
  return (b >> 63) ? -(long long)v : (long long)v;
}

// s 2^-62 as a float64, rounded to nearest, for s > 0
IM_FN double unit62_to_double(long long s) {
  const int lz = __clzll(s);
  const unsigned long long n = (unsigned long long)s << lz;
  const unsigned long long m = (n >> 11) + ((n >> 10) & 1ULL);
  return __longlong_as_double((long long)(m + ((unsigned long long)(1023 - lz) << 52)));
}

// one Horner step s <- c + s x, s and c of unit 2^-62, x of unit 2^-66
IM_FN long long horner62(long long s, long long x, long long c) { return c + (__mul64hi(s, x) >> 2); }

constexpr long long U62(double v) { return (long long)(v * 4611686018427387904.0); }  // 2^62

// P(x) = (x - log1p x)/x^2 = 1/2 - x/3 + x^2/4 - ..., |x| < 2^-5: terms 0 to 5
// in 64-bit fixed point, 6 to 10 (below 2^-30 of the sum) in float32
IM_FN double log1p_tail(double x) {
  const long long f = small_to_fixed(x);
  const float y = __int2float_rn((int)(f >> 32)) * 0x1p-34f;
  const float t = 1.0f / 8 + y * (-1.0f / 9 + y * (1.0f / 10 + y * (-1.0f / 11 + y * (1.0f / 12))));
  long long s = (long long)__float2int_rn(t * 0x1p30f) << 32;
  s = horner62(s, f, U62(-1.0 / 7));
  s = horner62(s, f, U62(1.0 / 6));
  s = horner62(s, f, U62(-1.0 / 5));
  s = horner62(s, f, U62(1.0 / 4));
  s = horner62(s, f, -0x1555555555555555LL);  // 1/3
  s = horner62(s, f, 1LL << 61);
  return unit62_to_double(s);
}

// Q(x) = (expm1 x - x)/x^2 = 1/2 + x/6 + x^2/24 + ..., |x| < 2^-4: terms 0 to 4
// in 64-bit fixed point, 5 to 8 (below 2^-32 of the sum) in float32
IM_FN double expm1_tail(double x) {
  const long long f = small_to_fixed(x);
  const float y = __int2float_rn((int)(f >> 32)) * 0x1p-34f;
  const float t = 1.0f / 5040 + y * (1.0f / 40320 + y * (1.0f / 362880 + y * (1.0f / 3628800)));
  long long s = (long long)__float2int_rn(t * 0x1p42f) << 20;  // t < 2^-12
  s = horner62(s, f, U62(1.0 / 720));
  s = horner62(s, f, U62(1.0 / 120));
  s = horner62(s, f, U62(1.0 / 24));
  s = horner62(s, f, 0x0AAAAAAAAAAAAAAALL);  // 1/6
  s = horner62(s, f, 1LL << 61);
  return unit62_to_double(s);
}

// q(u) = 1 + u/3 + u^2/5 + ... (atanh(x)/x, u = x^2) and its reciprocal for
// 0 <= u < 1e-2 in fixed point: terms 0 to 4 in 64 bits, 5 to 8 (below 2^-36
// of the sum) in float32; ~65 integer instructions each instead of 8 float64
// ones and a division
IM_FN double atanhc(long long x) {
  const float y = __int2float_rn((int)(x >> 32)) * 0x1p-34f;
  const float t = 1.0f / 11 + y * (1.0f / 13 + y * (1.0f / 15 + y * (1.0f / 17)));
  long long s = (long long)__float2int_rn(t * 0x1p30f) << 32;
  s = horner62(s, x, U62(1.0 / 9));
  s = horner62(s, x, U62(1.0 / 7));
  s = horner62(s, x, U62(1.0 / 5));
  s = horner62(s, x, 0x1555555555555555LL);  // 1/3
  s = horner62(s, x, 1LL << 62);
  return unit62_to_double(s);
}

IM_FN double inv_atanhc(long long x) {
  const float y = __int2float_rn((int)(x >> 32)) * 0x1p-34f;
  const float t = -0.021796804f + y * (-0.016787552f + y * (-0.013502765f + y * -0.011203746f));
  long long s = (long long)__float2int_rn(t * 0x1p32f) << 30;
  s = horner62(s, x, U62(-428.0 / 14175.0));
  s = horner62(s, x, U62(-44.0 / 945.0));
  s = horner62(s, x, U62(-4.0 / 45.0));
  s = horner62(s, x, -0x1555555555555555LL);
  s = horner62(s, x, 1LL << 62);
  return unit62_to_double(s);
}

// X 2^-unit as a float64, rounded to nearest (ties away from zero)
template <int UNIT_ = UNIT>
IM_FN double to_double(long long X) {
  const unsigned long long u = (unsigned long long)(X < 0 ? -X : X);
  const int lz = __clzll((long long)u);
  const unsigned long long n = u << (lz & 63);
  const unsigned long long m = (n >> 11) + ((n >> 10) & 1ULL);
  const unsigned long long b = u ? m + ((unsigned long long)(1023 + 63 - UNIT_ - lz - 1) << 52) : 0ULL;
  return __longlong_as_double((long long)(b | (X < 0 ? 0x8000000000000000ULL : 0ULL)));
}

// x in units of 2^-57, rounded to nearest; false for |x| >= 64 (and NaN)
IM_FN bool from_double(double x, long long& X) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  const int e = (int)(b >> 52) & 0x7ff;
  if (e >= 1023 + 6) return false;
  const unsigned long long M = (b & 0xFFFFFFFFFFFFFULL) | 0x10000000000000ULL;
  // x = M 2^(e - 1075): X = M 2^(e - 1075 + 57)
  const int s = e - (1075 - UNIT);
  const unsigned long long v = s >= 0 ? M << s : (s < -60 ? 0ULL : ((M >> (-s - 1)) + 1ULL) >> 1);
  X = (b >> 63) ? -(long long)v : (long long)v;
  return true;
}

}  // namespace im
}  // namespace esplit
