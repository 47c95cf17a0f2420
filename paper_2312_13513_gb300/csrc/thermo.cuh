// Mixture thermodynamics of one cell from the NASA-7 coefficients of the mechanism blob (device
// code shared by the surrogate's post-processing and the thermo kernels).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "chem_internal.h"
#include "fixed.cuh"

namespace chem {

// Species enthalpies and heat capacities in fixed point (FxEnthalpy): five multiply-highs a
// polynomial on the integer pipe where the FP64 form takes five to seven FP64 instructions.
// Temperatures in [kTlo, kThi); outside, the callers use the FP64 polynomials.
struct Tau {
  fx::u64 t;
  fx::i64 t2;
  float tf;
  int rg;
  bool fast;
};
__device__ __forceinline__ Tau tau_of(double T) {
  Tau q;
  q.fast = (unsigned)__double2hiint(T) - 0x40600000u < 0x40b00000u - 0x40600000u;
  int e;
  const fx::u64 m = fx::mantissa(q.fast ? T : 1024.0, e);
  q.rg = __double2hiint(T) < 0x408f4000 ? 0 : 1;               // T < 1000, for T > 0
  q.t = m >> (((q.fast && q.rg == 0) ? kFxR0 - 1 : kFxR1 - 1) - e);
  q.t2 = (fx::i64)(q.t >> 1);
  q.tf = (float)(unsigned)(q.t >> 32) * 2.3283064365386963e-10f;
  return q;
}
// one value of a table in global (read-only) or, SH, shared memory
template <bool SH, class V> __device__ __forceinline__ V tab_ld(const V* p) {
  if constexpr (SH) return *p;
  else return __ldg(p);
}
// h/(R W) of a species
template <bool SH = false>
__device__ __forceinline__ double fx_enthalpy(const FxEnthalpy& E, const Tau& q) {
  const fx::u64 B = 0x8000000000000000ull;
  fx::u64 a = (fx::u64)tab_ld<SH>((const long long*)&E.h[5]);
#pragma unroll
  for (int i = 4; i >= 0; --i)
    a = (fx::umulhi3(a, q.t) + (fx::u64)(tab_ld<SH>((const long long*)&E.h[i]) - q.t2)) ^ (i ? B : 0ull);
  return fx::to_double((fx::i64)a, tab_ld<SH>(&E.fh));
}
// cp/(R W) of a species
__device__ __forceinline__ double fx_cp(const FxEnthalpy& E, const Tau& q) {
  const fx::u64 B = 0x8000000000000000ull;
  fx::u64 a = (fx::u64)__ldg((const long long*)&E.c[4]);
#pragma unroll
  for (int i = 3; i >= 0; --i)
    a = (fx::umulhi3(a, q.t) + (fx::u64)(__ldg((const long long*)&E.c[i]) - q.t2)) ^ (i ? B : 0ull);
  return fx::to_double((fx::i64)a, __ldg(&E.fc));
}
// cp/(R W) in FP32, for Newton steps on T (it scales the step, not the result)
template <bool SH = false>
__device__ __forceinline__ float cp_f32(const FxEnthalpy& E, const Tau& q) {
  float r = tab_ld<SH>(&E.cf[4]);
#pragma unroll
  for (int i = 3; i >= 0; --i) r = fmaf(q.tf, r, tab_ld<SH>(&E.cf[i]));
  return r;
}
// Order of doubles by their bit patterns (an FP64 compare takes the FP64 pipe as long as an FMA):
// |a| < |b|, with NaN above infinity; lo <= x <= hi for positive bounds, false for NaN
__device__ __forceinline__ bool less_abs(double a, double b) {
  const long long M = 0x7fffffffffffffffll;
  return (__double_as_longlong(a) & M) < (__double_as_longlong(b) & M);
}
__device__ __forceinline__ bool in_bounds(double x, double lo, double hi) {
  const long long b = __double_as_longlong(x);
  return b >= __double_as_longlong(lo) && b <= __double_as_longlong(hi);
}

// FP32 value near x (truncated; zero below the normal range) and exact FP64 value of f without the
// FP64 pipe's conversion instructions (each takes the pipe as long as an FMA): the exponent is
// rebiased and the mantissa shifted by integer instructions
__device__ __forceinline__ float f32_of(double x) {
  const unsigned h = (unsigned)__double2hiint(x), e = h & 0x7ff00000u;
  if (e < 0x38100000u) return 0.0f;
  if (e >= 0x47e00000u) return (float)x;
  const unsigned m = __funnelshift_l((unsigned)__double2loint(x), h, 3);
  return __uint_as_float((h & 0x80000000u) | ((m - 0xC0000000u) & 0x7fffffffu));
}
__device__ __forceinline__ double f64_of(float f) {
  const unsigned u = __float_as_uint(f), e = u & 0x7f800000u;
  if (e == 0u) return (u & 0x7fffffffu) ? (double)f : __hiloint2double((int)u, 0);
  if (e == 0x7f800000u) return (double)f;
  return __hiloint2double((int)((u & 0x80000000u) | (((u & 0x7fffffffu) >> 3) + 0x38000000u)), (int)(u << 29));
}

// Mass-specific enthalpy h (erg/g, formation included) and cp (erg/(g K)) at temperature T of
// the composition Yloc[k] (if given) or Y[k * ld + cell].
__device__ __forceinline__ void h_cp_mass(const unsigned char* blob, const MechLayout& L, double T,
                                          const double* Y, int64_t ld, int64_t cell, const double* Yloc,
                                          double* h, double* cp) {
  const int ns = L.ns;
  const int rg = T < TMID ? 0 : 1;
  const double* hc = (const double*)(blob + L.o_hc);
  const double* cc = (const double*)(blob + L.o_cpc);
  const double* invW = (const double*)(blob + L.o_invW);
  const double invT = 1.0 / T;
  double hs = 0.0, cs = 0.0;
  for (int k = 0; k < ns; ++k) {
    const double* a = hc + (rg * ns + k) * 6;
    const double* c = cc + (rg * ns + k) * 5;
    const double hRT = a[0] + T * (a[1] + T * (a[2] + T * (a[3] + T * a[4]))) + a[5] * invT;
    const double cpR = c[0] + T * (c[1] + T * (c[2] + T * (c[3] + T * c[4])));
    const double yk = Yloc ? Yloc[k] : Y[k * ld + cell];
    hs += yk * hRT * __ldg(invW + k);
    cs += yk * cpR * __ldg(invW + k);
  }
  *h = RU * T * hs;
  *cp = RU * cs;
}

// Mass-specific enthalpy alone (erg/g, formation included) of the composition Yloc at T, as the
// polynomial h / R = a5 + a0 T + a1 T^2 + ... + a4 T^5 per species (no division by T).
__device__ __forceinline__ double h_mass(const unsigned char* blob, const MechLayout& L, double T,
                                         const double* Yloc) {
  const int ns = L.ns;
  const int rg = T < TMID ? 0 : 1;
  const double* hc = (const double*)(blob + L.o_hc);
  const double* invW = (const double*)(blob + L.o_invW);
  double hs = 0.0;
  for (int k = 0; k < ns; ++k) {
    const double* a = hc + (rg * ns + k) * 6;
    const double hR = a[5] + T * (a[0] + T * (a[1] + T * (a[2] + T * (a[3] + T * a[4]))));
    hs += Yloc[k] * hR * __ldg(invW + k);
  }
  return RU * hs;
}

// The mixture's NASA-7 polynomials for one temperature range: for mass fractions Yloc,
// Ah[i] = sum_k Y_k / W_k a_ik (the h/RT coefficients, a6 included) and Ac[i] likewise for cp/R,
// so that h = R T (Ah0 + Ah1 T + ... + Ah4 T^4 + Ah5 / T) and cp = R (Ac0 + ... + Ac4 T^4): a
// Newton iteration on T at fixed composition then costs one polynomial instead of one per
// species (the same sums, reordered).
__device__ __forceinline__ void mixture_nasa(const unsigned char* blob, const MechLayout& L, int rg,
                                             const double* Yloc, double Ah[6], double Ac[5]) {
  const int ns = L.ns;
  const double* hc = (const double*)(blob + L.o_hc);
  const double* cc = (const double*)(blob + L.o_cpc);
  const double* invW = (const double*)(blob + L.o_invW);
  for (int i = 0; i < 6; ++i) Ah[i] = 0.0;
  for (int i = 0; i < 5; ++i) Ac[i] = 0.0;
  for (int k = 0; k < ns; ++k) {
    const double yw = Yloc[k] * __ldg(invW + k);
    const double* a = hc + (rg * ns + k) * 6;
    const double* c = cc + (rg * ns + k) * 5;
    for (int i = 0; i < 6; ++i) Ah[i] = fma(yw, a[i], Ah[i]);
    for (int i = 0; i < 5; ++i) Ac[i] = fma(yw, c[i], Ac[i]);
  }
}

// h and cp of a mixture polynomial at T; h = R (Ah5 + Ah0 T + ... + Ah4 T^5), no division by T
__device__ __forceinline__ void h_cp_from_mixture(const double Ah[6], const double Ac[5], double T, double* h,
                                                  double* cp) {
  *h = RU * (Ah[5] + T * (Ah[0] + T * (Ah[1] + T * (Ah[2] + T * (Ah[3] + T * Ah[4])))));
  *cp = RU * (Ac[0] + T * (Ac[1] + T * (Ac[2] + T * (Ac[3] + T * Ac[4]))));
}

}  // namespace chem
