// Float64 z derivatives by the dense operators in exact integer arithmetic:
// number formats, index maps and the exact continuation, shared by the kernel
// (k_dense64.cu), the table builder and the CPU checks.
//
// A line is brought to whole numbers of 2^(E - 1082), E the exponent of its
// largest value (|x| < 2^60; with 2^53, a line with a peak lost up to 3.6 times
// what the transform loses), split into its NQ parts (dense_geom.hpp; |u| <
// 2^62, exact) and every part into eight balanced base-256 digits.  The
// operators' blocks are whole numbers of 2^-e below 2^63 (rounded once, from
// binary128; with 2^55, twice the transform's error), in eight digits.  Digits are exact in
// float16, and a sum of digit products stays a whole number below 2^24 (the
// CPU tests check the bound for every N'), so the tensor cores add them up exactly in
// float32.  Digit products of one weight share an accumulator: the eight
// leading weights are kept (36 of 64 products), what is left out is about 2^-56
// of the largest entry times the largest value.
#pragma once
#include <cstdint>

#include "dense_geom.hpp"

namespace fcns {

constexpr int kD64Lines = 16;    // lines per tile: the rows of one matrix instruction
constexpr int kD64Digits = 8;
constexpr int kD64Sums = 8;      // weights kept: digits i of the line and j of the operator with i + j < 8

// dense_geom for float64: both orders' blocks take 2.65 MB at most (they are read once per tile)
inline bool dense64_geom(int Nz, int Np, DenseGeom* o) {
  DenseGeom g;
  if (!dense_geom(Nz, Np, &g) || (g.NQ == 2 && g.KQ > 192)) return false;
  *o = g;
  return true;
}
FC_DG long long dense64_order_halves(const DenseGeom& g) {
  return (long long)(g.KQ / 16) * g.NQ * (g.KQ / 16) * kD64Digits * 32 * 8;
}
// operand fragments of the 16 x 8 x 16 matrix instruction: lane and half of
// element (row, k) of A (8 halves per lane) and of (k, column) of two adjacent B (8 halves per lane)
FC_DG int d64_a_index(int row, int k) { return ((row & 7) * 4 + (k & 7) / 2) * 8 + ((row >> 3) + 2 * (k >> 3)) * 2 + (k & 1); }
FC_DG int d64_b_index(int k, int col) { return ((col & 7) * 4 + (k & 7) / 2) * 8 + (2 * (col >> 3) + (k >> 3)) * 2 + (k & 1); }

// double (its bits) in whole units of 2^(E - 1082), rounded; E >= its exponent field
FC_DG long long d64_fixed(unsigned long long b, int E) {
  const int e = (int)(b >> 52) & 0x7ff;
  const unsigned long long m = (b & 0xfffffffffffffull) | (e ? 1ull << 52 : 0);
  const int s = E - (e ? e : 1);
  const long long v = s <= 7 ? (long long)(m << (7 - s)) : (s > 61 ? 0 : (long long)((m + (1ull << (s - 8))) >> (s - 7)));
  return b >> 63 ? -v : v;
}
// the digits as fields: digit i = field i - 128, field 0 the leading one
FC_DG unsigned long long d64_bias(long long u) { return (unsigned long long)u + 0x8080808080808080ull; }
FC_DG int d64_field(unsigned long long w, int i) { return (int)(w >> (8 * (7 - i))) & 255; }
// the eight sums (the first the heaviest) as one whole number, in units of 2^(56 + sh) of the product
// (modulo 2^64: the sum over the parts fits again)
FC_DG long long d64_combine(const int* a, int sh) {
  const long long hi = ((long long)a[0] << 24) + ((long long)a[1] << 16) + ((long long)a[2] << 8) + a[3];
  const long long lo = ((long long)a[4] << 24) + ((long long)a[5] << 16) + ((long long)a[6] << 8) + a[7];
  return (long long)(((unsigned long long)hi << (32 - sh)) + (unsigned long long)((lo + ((1ll << sh) >> 1)) >> sh));
}

FC_DG int d64_clz(unsigned long long v) {
#if defined(__CUDA_ARCH__)
  return __clzll((long long)v);
#else
  return v ? __builtin_clzll(v) : 64;
#endif
}

// C continuation value jj of a line (bits of its first d and last d values, `st`
// apart), the sum of the products exactly (to 2^-120 of the largest), rounded
// once: integer arithmetic, the float64 pipe being 1/74 of the integer one.
FC_DG unsigned long long d64_continuation(int jj, int d, int Cc, const double* Mr, const unsigned long long* first,
                                          const unsigned long long* last, int st) {
  int Emax = 0;
  __int128 acc = 0;
  for (int pass = 0; pass < 2; ++pass)
    for (int t = 0; t < 2 * d; ++t) {
      const int i = t < d ? t : t - d;
      const unsigned long long x = t < d ? last[i * st] : first[i * st];
      union { double v; unsigned long long b; } mr;
      mr.v = t < d ? Mr[jj * d + i] : Mr[(Cc - 1 - jj) * d + (d - 1 - i)];
      const int ex = (int)(x >> 52) & 0x7ff, em = (int)(mr.b >> 52) & 0x7ff;
      const unsigned long long mx = (x & 0xfffffffffffffull) | (ex ? 1ull << 52 : 0);
      const unsigned long long mm = (mr.b & 0xfffffffffffffull) | (em ? 1ull << 52 : 0);
      if (!mx || !mm) continue;
      const int e = (ex ? ex : 1) + (em ? em : 1);
      if (pass == 0) {
        if (e > Emax) Emax = e;
        continue;
      }
      const int s = Emax - e;
      if (s > 122) continue;
      const __int128 p = (__int128)((((unsigned __int128)mx * mm) << 16) >> s);   // < 2^122
      acc += (x ^ mr.b) >> 63 ? -p : p;
    }
  if (acc == 0) return 0;
  const unsigned long long sign = acc < 0 ? 1ull << 63 : 0;
  unsigned __int128 mag = acc < 0 ? (unsigned __int128)-acc : (unsigned __int128)acc;
  const unsigned long long h = (unsigned long long)(mag >> 64);
  const int lz = h ? d64_clz(h) : 64 + d64_clz((unsigned long long)mag);
  mag <<= lz;                                     // value = mag 2^(Emax - 16 - 2150 - lz)
  const unsigned long long top = (unsigned long long)(mag >> 64);   // 64 leading bits; 53 are kept
  const int e = Emax - 16 - 2150 - lz + 75 + 1075;   // exponent field of the result
  if (e >= 0x7ff) return sign | 0x7ff0000000000000ull;
  const int drop = e >= 1 ? 11 : 12 - e;          // a subnormal result keeps fewer bits
  if (drop > 63) return sign;
  const unsigned long long r = (top >> drop) + ((top >> (drop - 1)) & 1);
  return sign | (e >= 1 ? ((unsigned long long)(e - 1) << 52) + r : r);
}

}  // namespace fcns
