// ozslice.cuh -- FP64 values as balanced base-256 digits in BF16 slices, and sums of
// their products back to FP64 (error-free splitting; k_ozpotrf.cu, k_grad.cu).
#pragma once
#include "kernels.h"

namespace jmg {
namespace ozf {
constexpr int S = 7;            // slices per operand

// Which rows the slices stand in for.  A row (or column) is cut against its largest
// element, so an entry far below it keeps few digits or none, and a product of two rows
// whose large entries never meet would lose what an FMA keeps.  A row is FLAT when at
// least 9/16 of its entries lie within 4 binary exponents of its largest one: two flat
// rows p, q of length K then share K / 8 indices where |p_k q_k| > 2^-10 max|p| max|q|,
// so sum |p_k q_k| > 2^-13 K max|p| max|q|, and the error of the slices (about 2^-56
// sqrt(K) max|p| max|q|) stays at the level of the rounding of that sum, as FMAs' does.
// Everything else -- decaying, sparse and graded rows, and rows that are not finite --
// is SPREAD, and its products are formed with FP64 FMAs.  (Rows of the factors of matrices
// with dense eigenvectors, of Wishart factors and of solves with them are flat without
// exception; with 3 exponents in place of 4, one row in 2000 was not.)
constexpr int NEAR = 4;
JMG_DEV unsigned long long abs_bits(double x) {
  return (unsigned long long)__double_as_longlong(x) & 0x7FFFFFFFFFFFFFFFull;
}
__host__ __device__ constexpr int flat_count(int kv) { return (9 * kv + 15) / 16; }
// is |x| (its bits) within NEAR exponents of the row's maximum (mb)?
JMG_DEV bool near_max(unsigned long long b, unsigned long long mb) {
  return (int)(b >> 52) + NEAR >= (int)(mb >> 52);
}

// exponent e with |x| 2^-e < 1 for every |x| <= m (m as the bits of |x|);
// 0 for m == 0, infinities and NaN
JMG_DEV int scale_exp_bits(unsigned long long mb) {
  if (mb == 0) return 0;
  const int ex = (int)(mb >> 52);
  if (ex >= 0x7FF) return 0;
  if (ex) return ex - 1022;
  return -1010 - __clzll((long long)mb);  // subnormal: m = mb 2^-1074, mb < 2^(64-clz)
}

// A row's word: the exponent of its maximum mb in bits 0-15, the number of entries near it
// in bits 16-25 (none where no exponent lies below the maximum's by NEAR, nor in a row that
// is not finite); k_oz_strip counts the 64-column chunks that have added theirs from bit 26.
JMG_DEV bool can_be_flat(unsigned long long mb) {
  const int ex = (int)(mb >> 52);
  return mb == 0 || (ex > NEAR && ex < 0x7FF);
}
JMG_DEV int row_word(unsigned long long mb, int cnt) {
  const int e = scale_exp_bits(mb);
  return (e & 0xFFFF) | (can_be_flat(mb) ? cnt << 16 : 0);
}
JMG_DEV int word_exp(int w) { return (int)(short)w; }
JMG_DEV bool word_spread(int w, int flat) { return (w >> 16 & 1023) < flat; }

// The digits of x 2^-e (|x 2^-e| < 1): V = rint(x 2^(55-e)), |V| <= 2^55, cut into
// balanced base-256 digits from the bottom; integer operations only.
JMG_DEV void digits7(double x, int e, int (&d)[S]) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(x);
  int ex = (int)((b >> 52) & 0x7FF);
  unsigned long long M = b & ((1ull << 52) - 1);
  if (ex)
    M |= 1ull << 52;
  else
    ex = 1;
  const int sh = ex - 1020 - e;  // V = M 2^sh
  unsigned long long V = 0;
  if (sh >= 0) {
    V = sh <= 60 ? M << sh : 0ull;  // (below 2^55 for every finite row; subnormals shift far)
  } else if (sh > -64) {
    const int k = -sh;
    V = (M >> k) + ((M >> (k - 1)) & 1ull);  // to nearest, ties away
  }
  long long W = (b >> 63) ? -(long long)V : (long long)V;
#pragma unroll
  for (int s = S - 1; s >= 1; --s) {
    const int k = (int)(signed char)(W & 255);
    d[s] = k;
    W = (W - k) >> 8;
  }
  d[0] = (int)W;  // |W| <= 128
}

// v 2^ex rounded once to FP64 (to nearest even), in integer operations: a
// conversion holds the FP64 pipe as long as an FMA.
JMG_DEV double scaled_double(long long v, int ex) {
  if (v == 0) return 0.0;
  const unsigned long long u = v < 0 ? 0ull - (unsigned long long)v : (unsigned long long)v;
  const int lz = __clzll((long long)u);
  const unsigned long long m = u << lz;  // leading bit at 63
  const int E = 1086 - lz + ex;          // exponent field
  if (E < 1 || E > 2045) return ldexp((double)v, ex);
  unsigned long long q = m >> 11;
  const unsigned rem = (unsigned)m & 0x7FFu;
  q += (rem > 0x400u || (rem == 0x400u && (q & 1))) ? 1 : 0;
  // (a carry out of the significand moves into the exponent)
  const unsigned long long bits = ((unsigned long long)(E - 1) << 52) + q;
  return __longlong_as_double((long long)(bits | ((unsigned long long)v & (1ull << 63))));
}
}  // namespace ozf
}  // namespace jmg
