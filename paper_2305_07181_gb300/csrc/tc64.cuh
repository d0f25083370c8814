// Float64 operator contractions  out[c][m] = sum_n D_i[m][n] x[c][n]  of one
// element on the fp16 tensor cores, by error-free slicing (the integer form of
// the Ozaki scheme: Ozaki, Ogita, Oishi and Rump, Numer. Algorithms 59, 2012).
//
// What bounds it, and why: the float64 pipe of GB300 runs 1.68 FMAs per clock
// and SM, one warp instruction in ~19 clocks, while everything else (integer,
// float32, warp-level tensor instructions) runs 40 to 1000 times faster.  A
// float64 FMA loop over the operators therefore spends ~3/4 of the volume
// kernel on the contractions.  Here they take no float64 instruction at all:
//   * every row of D_i and every column of x becomes fixed point: a signed
//     integer of DIGITS BITS bits times a power of two taken from the row's or
//     the column's largest entry, cut into signed digits of BITS bits, each
//     exact in fp16 (digits.h);
//   * products of digits are sums of integers below 2^24, exact in the float32
//     accumulators of mma.sync (m16n8k16); digit pairs (j, a) of one weight
//     level j + a share accumulators;
//   * the levels are added up as 64-bit integers and rounded once to float64.
// Digits: six of 10 bits up to 32 nodes; above, where three digit products of
// 2^18 over 80 nodes would pass 2^24, seven of 9 bits.
//
// Accuracy, with A and X the powers of two above the largest entry of the row
// and of the column and u = 2^-53:
//   six digits:   |error| <= 2^-60 (X sum|D| + A sum|x|) + (n_p 2^-59 + 2^-56) A X + u |result|
//   seven digits: |error| <= 2^-63 (X sum|D| + A sum|x|) + (n_p 2^-60 + 2^-60) A X + 1.25 u |result|
// (quantisation of the operands; digit pairs left out: (2, 4), (4, 2) and all
// of level 7 on, or level 7 on; the last unit of the integer sum).  An FMA loop
// errs by the row's own summands instead, up to n_p u sum|D||x|.  So the sum
// here is the closer one as long as the products of a row reach a fair part of
// A X, and the loop is where a column's large entries meet only small entries
// of the row.  Measured against exact sums with the library's operators, in
// units of u sum|D||x|, root mean square (loop | here), one entry of the
// column larger than the others by the factor:
//   18 nodes: 1 0.57 | 0.19, 50 0.77 | 0.42, 1e3 1.3 | 2.8, 1e6 1.7 | 490
//   58 nodes: 1 0.69 | 0.13, 50 1.06 | 0.19, 1e3 1.9 | 0.8, 1e6 2.2 | 270
//
// Tile: the 16 rows of the A operand are 8 columns of x times 2 consecutive
// digits, the 8 columns of the B operand 8 rows m of D_i, so both digits'
// accumulators of an output (c, m) sit in one thread.  12 products of a
// 16 x 8 x 16 tile cover the 22 digit pairs of six digits, 16 the 28 of seven
// (the pair of digit 6 holds digit 6 twice; the second one's level is not
// used).  D_i is stored in 60 or 63 bits, two entries in 16 bytes, digits laid
// out so that one shift-and-mask step gives the fp16 pair of a digit (half the
// bytes of pre-cut fp16 digits; the cutting hides behind the float64 pointwise
// work of the other blocks of the SM).
//
// Columns whose largest entry is below 2^-958 count as zero; a column or row
// with a non-finite entry gives NaN, as a sum over it would.
#pragma once

#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "digits.h"

namespace esplit {
namespace tc {

// ---------------------------------------------------------------------------
// packed operators: opsP[e][i][m][pair] (uint4) holds D_i[m][2 pair] and
// D_i[m][2 pair + 1] (in the upper halfwords) as pack_half lays them out.
// opsE[e][i][m]: the row's exponent.
// ---------------------------------------------------------------------------
// one thread per (element, direction, row); ops64: [e][d][n][m]
template <int BITS>
__global__ void build_packed_kernel(const double* __restrict__ ops64, int n_e, int d, int np,
                                    uint4* __restrict__ opsP, short* __restrict__ opsE) {
  const size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= (size_t)n_e * d * np) return;
  const size_t ei = idx / np;
  const int m = (int)(idx - ei * np);
  const double* op = ops64 + (ei * np) * np + m;
  unsigned mx = 0;
  for (int n = 0; n < np; ++n) mx = max(mx, (unsigned)__double2hiint(op[(size_t)n * np]) & 0x7FFFFFFFu);
  const int E = exp_of_max(mx);
  opsE[idx] = (short)E;
  const int pairs = pairs_for(np);
  uint4* out = opsP + idx * pairs;
  for (int p = 0; p < pairs; ++p) {
    uint4 a, b;
    pack_half<BITS>(fixed_fields<BITS>(op[(size_t)(2 * p) * np], E), a.x, a.y, a.z, a.w);
    const double v1 = 2 * p + 1 < np ? op[(size_t)(2 * p + 1) * np] : 0.0;
    pack_half<BITS>(fixed_fields<BITS>(v1, E), b.x, b.y, b.z, b.w);
    out[p] = make_uint4(a.x | (b.x << 16), a.y | (b.y << 16), a.z | (b.z << 16), a.w | (b.w << 16));
  }
}

template <int BITS>
__device__ __forceinline__ unsigned unbias(unsigned fields) {  // two 16-bit fields -> two fp16 digits
  constexpr unsigned MASK = BITS == 10 ? 0x03FF03FFu : 0x01FF01FFu;
  const unsigned h = (fields & MASK) | 0x64006400u;           // 1024 + field
  const unsigned c = BITS == 10 ? 0x66006600u : 0x65006500u;  // 1024 + 2^(BITS-1)
  unsigned r;
  asm("sub.rn.f16x2 %0, %1, %2;" : "=r"(r) : "r"(h), "r"(c));
  return r;
}

template <int BITS>
__device__ __forceinline__ void unpack(const uint4& q, unsigned (&s)[digits_of(BITS)]) {
  unpack_fields<BITS>(q.x, q.y, q.z, q.w, s);
#pragma unroll
  for (int k = 0; k < digits_of(BITS); ++k) s[k] = unbias<BITS>(s[k]);
}

__device__ __forceinline__ void mma16(float (&c)[4], const unsigned (&a)[4], unsigned b0, unsigned b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}

__device__ __forceinline__ void mma8(float (&c)[4], unsigned a0, unsigned a1, unsigned b0) {
  asm("mma.sync.aligned.m16n8k8.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5}, {%6}, {%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a0), "r"(a1), "r"(b0));
}

__device__ __forceinline__ void ldm4(unsigned (&r)[4], unsigned addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(addr)
               : "memory");
}

__device__ __forceinline__ void ldm2(unsigned& r0, unsigned& r1, unsigned addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x2.shared.b16 {%0,%1}, [%2];"
               : "=r"(r0), "=r"(r1)
               : "r"(addr)
               : "memory");
}

// Sizes of one block's contraction over EB elements of NP nodes.  Columns per
// element and direction: NF columns that differ by direction and whose results
// are summed over the directions (f_i -> sum_i D_i f_i), and NW columns shared
// by the directions, one result each (w -> D_i w).
template <int D, int NP, int EB, int NF, int NW, int THREADS>
struct Shape {
  static constexpr int BITS = bits_for(NP);
  static constexpr int DIGITS = digits_of(BITS);
  static constexpr int KP = (NP + 7) / 8 * 8;          // nodes padded to the tile
  static constexpr int K16 = KP / 16;                  // 16-node tiles, then one of 8 if KP % 16
  static constexpr bool K8 = KP % 16 != 0;
  static constexpr int NT = (NP + 7) / 8;              // tiles of 8 output rows
  // 32-bit words of a digit row: an odd multiple of 4, so that the eight rows
  // an ldmatrix reads fall in different banks
  static constexpr int NPW = (KP / 2) % 8 == 4 ? KP / 2 : KP / 2 + 4;
  static constexpr int COLS = D * NF + NW;             // distinct columns of x
  static constexpr int MB = (NF + NW + 7) / 8;         // row blocks of 8 columns per direction
  static constexpr int OUTS = NF + D * NW;             // results per node
  // row stride of the results (doubles): an odd multiple of 4 against bank
  // conflicts, except where the shorter row lets a sixth block on the SM
  static constexpr int NPO = NP == 18 ? 18 : (NP + 3) / 8 * 8 + 4;
  static constexpr int NPH = NP | 1;                   // row stride of the high words (odd)
  static constexpr int T = BITS == 10 ? 6 : 7;         // accumulator tiles
  // unit of the 64-bit level sums, 2^-UNIT of the digit products' unit: the
  // sum over NP nodes and D directions stays below 2^63
  static constexpr int UNIT = BITS == 10 ? (D == 3 ? 62 : 61) : 69;
  static constexpr size_t DIG_EL = (size_t)DIGITS * COLS * NPW * 4, RES_EL = (size_t)OUTS * NPO * 8;  // bytes per element
  // Where every warp takes the same number of an element's row tiles, the
  // element's results go over the digits of the element before it (a block
  // barrier between the elements), the first one's to a region of its own:
  // 53 instead of 71 KB per block at 25 nodes, four blocks per SM instead of
  // three (Navier-Stokes kernel, 24,576 tetrahedra: 780 -> 680 us); with seven
  // digits, 50 instead of 60 KB at 58 nodes and 63 instead of 76 KB at 78 (four
  // and three blocks instead of three and two; 3,072 and 1,296 tetrahedra: 181
  // -> 177 and 161 -> 143 us).  Six-digit blocks of fewer than four elements
  // are held to the same number by other limits.
  static constexpr bool OVER = EB >= (BITS == 10 ? 4 : 2) && NT % (THREADS / 32) == 0 && RES_EL <= DIG_EL;
  static constexpr size_t HI_BYTES = (size_t)EB * COLS * NPH * 4;  // the columns' high words, before the digits
  static constexpr size_t DIG_BYTES = EB * DIG_EL > HI_BYTES ? EB * DIG_EL : (HI_BYTES + 15) / 16 * 16;
  static constexpr size_t RES_BYTES = OVER ? RES_EL : EB * RES_EL;
  static __device__ __forceinline__ double* results(void* dig, double* res, int el) {
    if constexpr (OVER)
      return el == 0 ? res : reinterpret_cast<double*>(static_cast<unsigned char*>(dig) + (size_t)(el - 1) * DIG_EL);
    else
      return res + (size_t)el * OUTS * NPO;
  }
  static constexpr size_t EX_BYTES = (size_t)(EB * COLS + 3) / 4 * 16;
};

// v (COLS values of node m of element el) -> shared digit rows, with zero
// digits for the padding nodes (NP .. KP - 1).  Three steps with block barriers
// between them: high words out (in the digits' place), column maxima, digits.
// Every thread of the block calls it; `on`: the thread owns a node.
template <class S, int NP, int EB, int THREADS>
__device__ __forceinline__ void digitize(const double (&v)[S::COLS], bool on, int el, int m, int* ex, __half* dig) {
  constexpr int COLS = S::COLS;
  unsigned* hiw = reinterpret_cast<unsigned*>(dig);
  if (on) {
#pragma unroll
    for (int c = 0; c < COLS; ++c)
      hiw[(el * COLS + c) * S::NPH + m] = (unsigned)__double2hiint(v[c]) & 0x7FFFFFFFu;
  }
  __syncthreads();
  for (int j = threadIdx.x; j < EB * COLS; j += THREADS) {
    unsigned mx = 0;
#pragma unroll 6
    for (int n = 0; n < NP; ++n) mx = max(mx, hiw[j * S::NPH + n]);
    ex[j] = exp_of_max(mx);
  }
  __syncthreads();
  if constexpr (S::KP > NP) {
    constexpr int W = S::KP - NP;
    unsigned short* d = reinterpret_cast<unsigned short*>(dig);
    for (int j = threadIdx.x; j < EB * S::DIGITS * COLS * W; j += THREADS) {
      const int row = j / W, k = j - row * W;
      d[row * (2 * S::NPW) + NP + k] = 0;
    }
  }
  if (on) {
    unsigned short* row = reinterpret_cast<unsigned short*>(dig) + (size_t)el * S::DIGITS * COLS * (2 * S::NPW) + m;
    constexpr unsigned MASK = (1u << S::BITS) - 1u;
#pragma unroll
    for (int c = 0; c < COLS; ++c) {
      const unsigned long long b = fixed_fields<S::BITS>(v[c], ex[el * COLS + c]);
#pragma unroll
      for (int s = 0; s < S::DIGITS; s += 2) {
        constexpr int LAST = S::DIGITS - 1;
        const unsigned ua = (unsigned)(b >> ((LAST - s) * S::BITS)) & MASK;
        const unsigned ub = s < LAST ? (unsigned)(b >> ((LAST - 1 - s) * S::BITS)) & MASK : 0u;
        const unsigned h = unbias<S::BITS>(ua | (ub << 16));
        row[(s * COLS + c) * (2 * S::NPW)] = (unsigned short)h;
        if (s < LAST) row[((s + 1) * COLS + c) * (2 * S::NPW)] = (unsigned short)(h >> 16);
      }
    }
  }
}

// asks for bytes [p, p + n) in L2 (p and n multiples of 16): one request of the
// bulk-copy engine, issued before the pointwise phase whose ~10 us hide it
__device__ __forceinline__ void prefetch_l2(const void* p, unsigned n) {
  asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p), "r"(n) : "memory");
}

// The contraction of the block's elements: warps take (element, tile of 8
// rows) tasks, all directions each.  elems: element index of slot el or -1.
// Results: res[el][k][m], k < NF the sums over the directions, then
// NF + i NW + q for column q of direction i.
template <class S, int D, int NP, int EB, int NF, int NW, int THREADS>
__device__ __forceinline__ void contract(__half* dig, const int* ex, const int* elems,
                                         const uint4* __restrict__ opsP, const short* __restrict__ opsE, double* res) {
  constexpr int BITS = S::BITS, DIGITS = S::DIGITS, MB = S::MB, T = S::T, COLS = S::COLS;
  constexpr int PAIRS = pairs_for(NP);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int g = lane >> 2, t4 = lane & 3;
  const unsigned dig0 = (unsigned)__cvta_generic_to_shared(dig);
  // operator entries of one (task, direction): two loads per 16-node tile, one
  // for an 8-node tile; up to 32 nodes the next direction's (or task's) are
  // issued before the current one's digit sums are added up
  constexpr int NQ = 2 * S::K16 + (S::K8 ? 1 : 0);
  constexpr bool AHEAD = NP <= 32;
  auto fetch = [&](int task, int i, uint4 (&q)[NQ]) {
#pragma unroll
    for (int k = 0; k < NQ; ++k) q[k] = make_uint4(0u, 0u, 0u, 0u);
    if (task >= EB * S::NT) return;
    const int el = task / S::NT, mrow = (task - el * S::NT) * 8 + g, e = elems[el];
    if (e < 0 || mrow >= NP) return;
    const uint4* dp = opsP + (((size_t)e * D + i) * NP + mrow) * PAIRS;
#pragma unroll
    for (int k = 0; k < NQ; ++k)
      if (k * 4 + t4 < PAIRS) q[k] = __ldcs(&dp[k * 4 + t4]);
  };
  uint4 qn[NQ];
  if constexpr (AHEAD) fetch(warp, 0, qn);
  for (int task = warp; task < EB * S::NT; task += THREADS / 32) {
    const int el = task / S::NT, nt = task - el * S::NT;
    const int e = elems[el];
    double* out = S::results(dig, res, el);
    if (e >= 0) {                    // -1 only behind the last element of the list
    const int mo = nt * 8 + 2 * t4;  // first of the two rows of this lane's results
    long long fs[MB][2];
    int fE[MB][2];
#pragma unroll 1
    for (int i = 0; i < D; ++i) {
      const short* de = opsE + ((size_t)e * D + i) * NP;
      // ldmatrix row addresses: matrices 0, 2 hold digit 2a, 1, 3 digit 2a + 1
      // (where there is no digit 2a + 1, digit 2a again: `odd` taken off)
      const unsigned odd = (unsigned)((lane >> 3) & 1) * (COLS * S::NPW * 4);
      unsigned addr[MB];
#pragma unroll
      for (int mb = 0; mb < MB; ++mb) {
        int c = mb * 8 + (lane & 7);
        if (c >= NF + NW) c = NF + NW - 1;
        const int col = c < NF ? i * NF + c : D * NF + (c - NF);
        addr[mb] = dig0 + (((el * DIGITS) * COLS + col) * S::NPW) * 4 + odd + (lane >> 4) * 16;
      }
      float acc[MB][T][4];
#pragma unroll
      for (int mb = 0; mb < MB; ++mb)
#pragma unroll
        for (int k = 0; k < T; ++k)
#pragma unroll
          for (int r = 0; r < 4; ++r) acc[mb][k][r] = 0.0f;
      uint4 q[NQ];
      if constexpr (AHEAD) {
#pragma unroll
        for (int k = 0; k < NQ; ++k) q[k] = qn[k];
      } else {
        fetch(task, i, q);
      }
#pragma unroll
      for (int kt = 0; kt < S::K16; ++kt) {
        unsigned b0[DIGITS], b1[DIGITS];
        unpack<BITS>(q[2 * kt], b0);
        unpack<BITS>(q[2 * kt + 1], b1);
#pragma unroll
        for (int mb = 0; mb < MB; ++mb)
#pragma unroll
          for (int a = 0; a < (DIGITS + 1) / 2; ++a) {
            unsigned A[4];
            ldm4(A, addr[mb] - (2 * a + 1 < DIGITS ? 0u : odd) + (2 * a * COLS * S::NPW) * 4 + kt * 32);
#pragma unroll
            for (int j = 0; j < DIGITS; ++j)
              if (j + 2 * a < T) mma16(acc[mb][j + 2 * a], A, b0[j], b1[j]);
          }
      }
      if constexpr (S::K8) {
        constexpr int kt = S::K16;
        unsigned b0[DIGITS];
        unpack<BITS>(q[NQ - 1], b0);
#pragma unroll
        for (int mb = 0; mb < MB; ++mb)
#pragma unroll
          for (int a = 0; a < (DIGITS + 1) / 2; ++a) {
            unsigned A0, A1;
            ldm2(A0, A1, addr[mb] - (2 * a + 1 < DIGITS ? 0u : odd) - (lane >> 4) * 16 +
                             (2 * a * COLS * S::NPW) * 4 + kt * 32);
#pragma unroll
            for (int j = 0; j < DIGITS; ++j)
              if (j + 2 * a < T) mma8(acc[mb][j + 2 * a], A0, A1, b0[j]);
          }
      }
      if constexpr (AHEAD) fetch(i + 1 < D ? task : task + THREADS / 32, i + 1 < D ? i + 1 : 0, qn);
      // levels -> 64-bit sums -> float64, two rows of one column per lane
#pragma unroll
      for (int mb = 0; mb < MB; ++mb) {
        const int c = mb * 8 + g;
#pragma unroll
        for (int r = 0; r < 2; ++r) {
          float tt[T], bb[T];
#pragma unroll
          for (int k = 0; k < T; ++k) {
            tt[k] = acc[mb][k][r];
            bb[k] = acc[mb][k][2 + r];
          }
          int fine;
          long long J = level_sum<BITS, S::UNIT, NP, T>(tt, bb, fine);
          const int col = c < NF ? i * NF + c : D * NF + (c - NF);
          const bool live = c < NF + NW && mo + r < NP;
          int E = live ? ex[el * COLS + col] + (int)__ldg(&de[mo + r]) - fine : 0;
          if (NF > 0 && c < NF) {  // the sum over the directions so far
            if (i > 0) {
              add_direction(fs[mb][r], fE[mb][r], J, E);
              J = fs[mb][r];
              E = fE[mb][r];
            } else {
              fs[mb][r] = J;
              fE[mb][r] = E;
            }
          }
          if (live && (c >= NF || i == D - 1)) {
            const int k = c < NF ? c : NF + i * NW + (c - NF);
            out[k * S::NPO + mo + r] = level_value<BITS, S::UNIT>(J, E);
          }
        }
      }
    }
    }
    if constexpr (S::OVER) {
      // all warps are through with this element's digits before the next
      // element's results go there (uniform: OVER makes the counts equal)
      constexpr int PER = S::NT / (THREADS / 32);
      if ((task / (THREADS / 32) + 1) % PER == 0) __syncthreads();
    }
  }
}

}  // namespace tc
}  // namespace esplit
