// Exponentials, logarithms and reciprocals of the FP64 kernels on the integer pipe.
//
// What bounds these kernels on this GPU is the FP64 pipe: one FP64 warp instruction takes 19 SM
// cycles (64 on its sub-partition, 76 with all four busy), a 64-bit integer multiply-high 4.8 and
// a 32 x 32 -> 64 multiply 1.2 (measured).  The library's exp, log and log10 are 17, 30 and 32 FP64
// instructions, a division 4.5 to 9, the table-driven exp_tab ten.  Here the same functions run in
// 64-bit fixed point: exp2_q52 about 25 SM cycles in place of 190, log2 about 45 in place of 570.
//
// Formats (Qa.b: b fraction bits of a 64-bit word):
//   Q11.52 signed   base-2 logarithms (of rate constants, Gibbs energies): absolute error 2^-52, so
//                   an exponential of them is good to about one unit in the last place whatever
//                   the argument's size, where an FP64 argument x carries |x| half units of its own
//   Q4.60 unsigned  log2 T for T in [kTlo, kThi)
//   Q0.64 unsigned  kTlo / T and T / 2^r (polynomial variable)
// Methods: 2^x by a 256-entry table of 2^(j / 256) and the Taylor polynomial of the rest (after
// Tang, ACM TOMS 15(2), 1989); log2 m by a table of 7-bit reciprocals c and the Taylor series of
// log2(1 + r), r = m c - 1 formed exactly; 1 / m by Newton's iteration v <- v (2 - m v).
// The functions are plain integer arithmetic, compiled for the host too (checked there against
// long double over the whole range).
#pragma once
#include <stdint.h>

#include "fixed_tables.h"

#ifdef __CUDACC__
#define FX_FN __host__ __device__ __forceinline__
#else
#define FX_FN static inline
#endif

namespace chem {
namespace fx {

typedef unsigned long long u64;
typedef long long i64;

// temperatures the fixed-point path takes; outside, the callers use FP64 throughout
constexpr double kTlo = 128.0, kThi = 4096.0;
constexpr int kTloExp = 7;

FX_FN u64 umulhi(u64 a, u64 b) {
#ifdef __CUDA_ARCH__
  return __umul64hi(a, b);
#else
  return (u64)(((unsigned __int128)a * b) >> 64);
#endif
}
// umulhi from the three upper partial products only (the fractions of the middle ones dropped): at
// most two units low
FX_FN u64 umulhi3(u64 a, u64 b) {
  const uint32_t al = (uint32_t)a, ah = (uint32_t)(a >> 32), bl = (uint32_t)b, bh = (uint32_t)(b >> 32);
  return ((u64)ah * bh + (((u64)al * bh) >> 32)) + (((u64)ah * bl) >> 32);
}
// Signed times unsigned for a loop-invariant factor b: the signed operand carries a bias of 2^63
// (its sign bit flipped), a b 2^-64 = umulhi3(biased a, b) - b / 2, and the caller folds the
// constant b / 2 into the next addition.
FX_FN u64 biased(i64 a) { return (u64)a ^ 0x8000000000000000ull; }
FX_FN uint32_t umulhi32(uint32_t a, uint32_t b) { return (uint32_t)(((u64)a * b) >> 32); }
// high word of signed a times unsigned b (floor)
FX_FN i64 mulhi_su(i64 a, u64 b) { return (i64)umulhi((u64)a, b) - (i64)((u64)(a >> 63) & b); }
FX_FN i64 mulhi_ss(i64 a, i64 b) {
#ifdef __CUDA_ARCH__
  return __mul64hi(a, b);
#else
  return (i64)(((__int128)a * b) >> 64);
#endif
}
FX_FN u64 bits_of(double x) {
#ifdef __CUDA_ARCH__
  return (u64)__double_as_longlong(x);
#else
  u64 b;
  __builtin_memcpy(&b, &x, 8);
  return b;
#endif
}
FX_FN double double_of(u64 b) {
#ifdef __CUDA_ARCH__
  return __longlong_as_double((i64)b);
#else
  double x;
  __builtin_memcpy(&x, &b, 8);
  return x;
#endif
}
FX_FN int clz64(u64 a) {
#ifdef __CUDA_ARCH__
  return __clzll((i64)a);
#else
  return a ? __builtin_clzll(a) : 64;
#endif
}

// nearest Q.52 of x, |x| < 2048 (the caller checks)
FX_FN i64 q52(double x) {
  const u64 b = bits_of(x);
  const int e = (int)((b >> 52) & 0x7ff) - 1023;            // |x| in [2^e, 2^(e+1))
  const u64 m = (b & 0x000fffffffffffffull) | 0x0010000000000000ull;
  u64 q;
  if (e >= 0) q = m << e;
  else q = e < -53 ? 0ull : (((m << 1) >> (-e)) + 1ull) >> 1;
  return (b >> 63) ? -(i64)q : (i64)q;
}

// x 2^-frac as the nearest double (ties up in magnitude)
FX_FN double to_double(i64 x, int frac) {
  if (x == 0) return 0.0;
  const u64 s = (u64)x & 0x8000000000000000ull;
  const u64 a = s ? (u64)(-x) : (u64)x;
  const int z = clz64(a);
  const u64 m = a << z;                                     // [2^63, 2^64)
  return double_of(s + ((u64)(1023 + 62 - z - frac) << 52) + (m >> 11) + ((m >> 10) & 1ull));
}

// 2^X for X in Q11.52, -1022 <= X < 1023 (the caller checks); tab: 256 mantissas of 2^(j / 256)
// times 2^62.  2^X = 2^n 2^(j/256) (1 + v): the terms above the second in 32 bits (they are below
// 2^-24 of the result), relative error below 2^-58 before the final rounding.
FX_FN double exp2_q52(i64 X, const u64* tab) {
  const u64 F = (u64)X << 20;                               // the fraction below 2^-8, times 2^72
  const uint32_t u = (uint32_t)(F >> 32);
  const uint32_t w3 = kE3 + umulhi32(u, kE4 + umulhi32(u, kE5));
  const u64 w2 = kE2 + (((u64)u * w3) >> 12);
  const u64 w1 = kE1 + (umulhi3(F, w2) >> 8);
  const u64 v = umulhi3(F, w1);                             // v 2^72
  const uint32_t xh = (uint32_t)((u64)X >> 32);
  const u64 t = tab[(xh >> 12) & 255u];
  const u64 m = ((t + 512ull) + (umulhi3(t, v) >> 8)) >> 10; // mantissa with its leading one at bit 52
  return double_of(m + ((u64)((xh & 0xfff00000u) + (1022u << 20)) << 32));
}
// X in the range of exp2_q52: one unsigned compare of the integer part
FX_FN bool exp2_in_range(i64 X) { return (uint32_t)((int)(X >> 52) + 1022) < 2045u; }

// log2 of a mantissa m in [1, 2) given as m 2^63, in Q.60 (modulo 2^64: a few units below zero at
// m = 1); rcp / lg: the 128-entry tables
FX_FN u64 log2_mant_q60(u64 m, const uint32_t* rcp, const u64* lg) {
  const uint32_t j = (uint32_t)(m >> 56) & 127u;
  const u64 c = rcp[j];
  // R = (m c - 1) 2^71 (m c 2^79 exactly in 80 bits; the one drops out modulo 2^64)
  const i64 R = (i64)((m * c >> 8) | (umulhi(m, c) << 56));
  i64 a = kL6 + (mulhi_ss(kL7, R) << 1);
  a = kL5 + (mulhi_ss(a, R) << 1);
  a = kL4 + (mulhi_ss(a, R) << 1);
  a = kL3 + (mulhi_ss(a, R) << 1);
  a = kL2 + (mulhi_ss(a, R) << 1);
  a = kL1 + (mulhi_ss(a, R) << 1);
  return lg[j] + (u64)(mulhi_ss(a, R) >> 9);                // 2^(70 + 63 - 64 - 9) = 2^60
}

// mantissa of a positive normal double times 2^63, and its exponent
FX_FN u64 mantissa(double x, int& e) {
  const u64 b = bits_of(x);
  e = (int)((b >> 52) & 0x7ff) - 1023;
  return ((b << 11) | 0x8000000000000000ull);
}

// log2 x in Q11.52 for a positive normal x
FX_FN i64 log2_q52(double x, const uint32_t* rcp, const u64* lg) {
  int e;
  const u64 m = mantissa(x, e);
  return ((i64)e << 52) + (i64)((log2_mant_q60(m, rcp, lg) + 128ull) >> 8);
}

// 2^63 / m for a mantissa m 2^63 in [1, 2), as a Q0.64 value in (1/2, 1): Newton's iteration in
// 64-bit integers from a 16-bit table value (16 -> 32 -> 64 bits; error a few units of 2^-64)
FX_FN u64 rcp_mant(u64 m, const uint32_t* rcp) {
  u64 v = ((u64)rcp[(uint32_t)(m >> 56) & 127u] << 48) - 1ull;            // 7-bit estimate, Q0.64
  // e = 1 - m v in Q.63 (|e| < 2^-7): m v = umulhi(m, v) 2^-63
  for (int it = 0; it < 4; ++it) {
    const i64 e = (i64)(0x8000000000000000ull - umulhi(m, v));
    v += (u64)(mulhi_su(e, v) << 1);
  }
  return v;
}

}  // namespace fx
}  // namespace chem
