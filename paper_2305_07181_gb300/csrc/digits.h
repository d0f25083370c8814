// Fixed-point digits of the tensor-core contraction (tc64.cuh): the integer
// arithmetic around the digit products, compiled for the device and, for the
// tests, for the host.
//
// A float64 x of a row or column whose largest entry is below 0.998 2^(E - 1022)
// becomes X = x 2^(1022 - E) 2^TOT rounded to an integer, TOT + 1 = DIGITS BITS
// bits, cut into DIGITS signed digits of BITS bits, each exact in fp16.
#pragma once

#include "imath.cuh"

namespace esplit {
namespace tc {

constexpr int NONFINITE = 1 << 14;  // exponent marker: the column or row holds an Inf or NaN

#ifdef __CUDACC__
#define DG_CONST __host__ __device__ constexpr
#else
#define DG_CONST constexpr
#endif
// 6 digits of 10 bits up to 32 nodes, 7 of 9 above
DG_CONST int bits_for(int np) { return np <= 32 ? 10 : 9; }
DG_CONST int digits_of(int bits) { return bits == 10 ? 6 : 7; }
DG_CONST int total_of(int bits) { return digits_of(bits) * bits - 1; }  // TOT: 59 or 62
DG_CONST int pairs_for(int np) { return (np + 1) / 2; }

// power-of-two exponent (biased, from the high words) of the largest entry:
// every entry is below 0.998 2^(E - 1022), within the signed digits' range
IM_FN int exp_of_max(unsigned hi_abs_max) {
  const int e = (int)((hi_abs_max + 0x1100u) >> 20);
  return hi_abs_max >= 0x7FF00000u ? NONFINITE : e;
}

// x as DIGITS unsigned BITS-bit fields (most significant first from bit TOT),
// field = digit + 2^(BITS-1), relative to the exponent E of exp_of_max
template <int BITS>
IM_FN unsigned long long fixed_fields(double x, int E) {
  constexpr int F = total_of(BITS) + 1;
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  const int e = (int)(b >> 52) & 0x7ff;
  const unsigned long long M = (b & 0xFFFFFFFFFFFFFULL) | 0x10000000000000ULL;
  constexpr int UP = F - 54;
  const int gap = E - e;
  const int d = E < 64 || gap > 63 ? 63 : gap;
  // right shift by d, rounded to nearest
  const unsigned long long v = (((M << (UP + 1)) >> (d & 63)) + 1ULL) >> 1;
  constexpr unsigned long long BIAS = (1ULL << (BITS - 1)) * (((1ULL << F) - 1ULL) / ((1ULL << BITS) - 1ULL));
  return (b >> 63) ? BIAS - v : BIAS + v;
}

// Storage of an operator entry: its fields in four halfwords (x, y, z, w).
//   BITS 10: x: digit 0, low 6 bits of digit 2 above it; y: digit 1, high bits
//            of digit 2; z, w: digits 3, 4 and 5 likewise.
//   BITS 9:  digits 0 to 3, and above them the low 7 bits of digits 4, 5, 6 in
//            x, y, z and their upper 2 bits in w (bits 9-10, 11-12, 13-14).
template <int BITS>
IM_FN void pack_half(unsigned long long b, unsigned& x, unsigned& y, unsigned& z, unsigned& w) {
  constexpr int D = digits_of(BITS);
  constexpr unsigned MASK = (1u << BITS) - 1u;
  unsigned u[7] = {};
  for (int k = 0; k < D; ++k) u[k] = (unsigned)(b >> ((D - 1 - k) * BITS)) & MASK;
  if (BITS == 10) {
    x = u[0] | ((u[2] & 63u) << 10);
    y = u[1] | ((u[2] >> 6) << 10);
    z = u[3] | ((u[5] & 63u) << 10);
    w = u[4] | ((u[5] >> 6) << 10);
  } else {
    x = u[0] | ((u[4] & 127u) << 9);
    y = u[1] | ((u[5] & 127u) << 9);
    z = u[2] | ((u[6] & 127u) << 9);
    w = u[3] | ((u[4] >> 7) << 9) | ((u[5] >> 7) << 11) | ((u[6] >> 7) << 13);
  }
}

// the fields of two packed entries (the second in the upper halfwords), one
// shift-and-mask step per digit; digits 0, 1, 3 and 4 (BITS 10), 0 to 3 (BITS 9)
// come unmasked
template <int BITS>
IM_FN void unpack_fields(unsigned x, unsigned y, unsigned z, unsigned w, unsigned (&f)[digits_of(BITS)]) {
  f[0] = x;
  f[1] = y;
  if constexpr (BITS == 10) {
    f[2] = ((x >> 10) & 0x003F003Fu) | ((y >> 4) & 0x03C003C0u);
    f[3] = z;
    f[4] = w;
    f[5] = ((z >> 10) & 0x003F003Fu) | ((w >> 4) & 0x03C003C0u);
  } else {
    f[2] = z;
    f[3] = w;
    f[4] = ((x >> 9) & 0x007F007Fu) | ((w >> 2) & 0x01800180u);
    f[5] = ((y >> 9) & 0x007F007Fu) | ((w >> 4) & 0x01800180u);
    f[6] = ((z >> 9) & 0x007F007Fu) | ((w >> 6) & 0x01800180u);
  }
}

// Sum of the weight levels of one output, in units of 2^(UNIT - fine) digit-
// product units: t[k], b[k] the accumulators of level k (even digit of x) and
// k + 1 (odd digit).  Integer sums of at most 2^24 convert exactly.
//   BITS 10 (NP <= 32): levels 0 to 3 exact, 4 to 6 to float32; fine = 0.
//   BITS 9: levels 0 to 5 exact (three pairs of 2^16 over 80 nodes), 6 to
//   float32; b[6], level 7, is left out.  UNIT = 69 keeps the largest sum of
//   three directions below 2^63, but it is 2^-55 of A X, the bound of one
//   product.  So sums below about A X (level 0 below 2^16; three of them stay
//   below 2^63) keep six more bits, fine = 6, and the unit is below 2^-54 of a
//   larger sum.
template <int BITS, int UNIT, int NP, int T>
IM_FN long long level_sum(const float (&t)[T], const float (&b)[T], int& fine) {
  // floats whose two parts may together exceed 2^24 are converted one by one
  const int i0 = __float2int_rn(t[0]);
  const int i1 = __float2int_rn(t[1] + b[0]);
  if constexpr (BITS == 10) {
    const int i2 = NP <= 21 ? __float2int_rn(t[2] + b[1]) : __float2int_rn(t[2]) + __float2int_rn(b[1]);
    const int i3 = __float2int_rn(t[3]) + __float2int_rn(b[2]);
    const float low = (t[4] + b[3]) + ((t[5] + b[4]) + b[5] * 0x1p-10f) * 0x1p-10f;
    const int il = __float2int_rn(low * (UNIT == 62 ? 0.25f : 0.5f));
    const long long hi = (long long)i0 * (1 << 20) + ((long long)i1 * (1 << 10) + i2);
    fine = 0;
    return (long long)((unsigned long long)hi << (80 - UNIT)) + ((long long)i3 * (1 << (70 - UNIT)) + il);
  } else {
    const int i2 = __float2int_rn(t[2] + b[1]);
    const int i3 = __float2int_rn(t[3]) + __float2int_rn(b[2]);
    const int i4 = __float2int_rn(t[4]) + __float2int_rn(b[3]);
    const float low = (t[5] + b[4]) + (t[6] + b[5]) * 0x1p-9f;
    fine = (unsigned)(i0 + 0xFFFF) < 0x1FFFFu ? 6 : 0;
    const int il = __float2int_rn(low * (fine ? 1.0f : 0x1p-6f));
    const long long hi = (long long)i0 * (1 << 18) + ((long long)i1 * (1 << 9) + i2);
    const unsigned long long up = ((unsigned long long)hi << 21) + ((unsigned long long)((long long)i3 * (1 << 12)) +
                                                                    (unsigned long long)((long long)i4 * 8));
    return (long long)(up << fine) + il;
  }
}

// adds the next direction's sum (J, E) to (S, ES), aligned to the larger exponent
IM_FN void add_direction(long long& S, int& ES, long long J, int E) {
  const int Em = E > ES ? E : ES, dj = Em - E, ds = Em - ES;
  S = (J >> (dj < 63 ? dj : 63)) + (S >> (ds < 63 ? ds : 63));
  ES = Em;
}

// v 2^(E - shift) rounded to nearest, E the sum of the two exponents of
// exp_of_max less level_sum's fine; NaN for a non-finite marker, zero below the
// normal range
template <int BITS, int UNIT>
IM_FN double level_value(long long v, int E) {
  // x = X 2^(Ex - 1022 - TOT): v has the unit 2^(UNIT - 2 TOT + E - 2044)
  constexpr int SH = UNIT - 2 * total_of(BITS) - 2044;
  const bool bad = E >= NONFINITE / 2;
  const unsigned sgn = (unsigned)((unsigned long long)v >> 63) << 31;
  const unsigned long long u = (unsigned long long)(v < 0 ? -v : v);
  const int lz = __clzll((long long)u);
  const unsigned long long n = u << (lz & 63);
  const unsigned long long r = (n >> 11) + ((n >> 10) & 1ULL);  // 53 bits, rounded (a carry goes to the exponent)
  const int ef = 63 - lz + 1023 + SH + E;                       // biased exponent
  unsigned long long bits = r + ((unsigned long long)(unsigned)(ef - 1) << 52);
  // overflow, underflow or a non-finite marker (from the largest exponent,
  // 2046, a carry of the rounding gives the bits of infinity by itself)
  if ((unsigned)(ef - 1) >= 2046u) {
    bits = ef > 0 ? 0x7FF0000000000000ULL : 0ULL;
    if (bad) bits = 0x7FF8000000000000ULL;
  }
  if (u == 0 && !bad) bits = 0ULL;
  return __longlong_as_double((long long)(bits | ((unsigned long long)sgn << 32)));
}

}  // namespace tc
}  // namespace esplit
