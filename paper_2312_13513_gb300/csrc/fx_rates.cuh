// Rate constants of the integrators from fixed-point base-2 exponents, with the FP64 forms for what
// lies outside the formats (fixed.cuh): shared by the cell-per-thread and the group kernels.
#pragma once

#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "chem_internal.h"
#include "fixed.cuh"

namespace chem {
namespace fx {

// tables of fixed.cuh, and the FP64 form of the mechanism in global memory
struct Ctx {
  const u64 *e2, *lg;
  const uint32_t* rc;
  const unsigned char* blob;
  const MechLayout* lay;
};

// 1 / x to about one unit in the last place in three FP64 instructions (the compiler's division
// takes 4.5 slots): the reciprocal approximation y (20 bits, on the special-function pipe), then
// y (1 + e + e^2) with e = 1 - x y, the third-order step of the geometric series, which leaves
// e^3 = 2^-60.  Arguments whose reciprocal would leave the normal range divide.
__device__ __forceinline__ double rcp(double x) {
  const unsigned hx = (unsigned)__double2hiint(x) & 0x7fffffffu;
  if (hx - 0x01000000u >= 0x7d000000u) return 1.0 / x;
  double y;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  const double e = fma(-x, y, 1.0);
  return fma(y, fma(e, e, e), y);
}

// larger of two non-negative doubles by their bit patterns (an FP64 compare is an FP64 slot)
__device__ __forceinline__ double max_pos(double a, double b) {
  return __double_as_longlong(a) > __double_as_longlong(b) ? a : b;
}

// exp(x): fixed point for |x| < 700, the library outside
__device__ __forceinline__ double exp_any(double x, const u64* e2) {
  const unsigned hx = (unsigned)__double2hiint(x) & 0x7fffffffu;
  if (hx >= 0x4085e000u) return (__double2hiint(x) < 0 && hx < 0x7ff00000u && hx >= 0x40900000u) ? 0.0 : exp(x);
  // x log2 e: |x| < 1024 in Q10.53 times log2 e in Q1.63, a Q11.52 product
  const i64 q = q52(x) * 2;
  return exp2_q52(mulhi_su(q, kLog2e), e2);
}

// log2 x as Q11.52 in range only: x positive, normal, finite (the caller's test)
__device__ __forceinline__ bool positive_normal(double x) {
  return (unsigned)__double2hiint(x) - 0x00100000u < 0x7ff00000u - 0x00100000u;
}

// Step-size factor 0.9 e^(-1/4) of an error norm e = sqrt(en2), at least 0.2; 0.2 for a non-finite
// norm.  2^(-log2(en2) / 8) in fixed point (sqrt and pow are 92 FP64 instructions).
__device__ __forceinline__ double step_factor(double en2, const u64* e2, const uint32_t* rc, const u64* lg) {
  if (((unsigned)__double2hiint(en2) & 0x7ff00000u) == 0x7ff00000u) return 0.2;
  if (!positive_normal(en2)) return 1e30;                  // en2 = 0: the caller's limit bounds it
  const i64 X = -(log2_q52(en2, rc, lg) >> 3);
  const double f = 0.9 * exp2_q52(X, e2);
  return f < 0.2 ? 0.2 : f;
}

// thermo state of a right-hand side at one temperature
struct Temp {
  double T, invT;
  u64 L, iT, tau;    // log2 T (Q4.60), 128 / T and T / 2^r (Q0.64); L and iT after slow_temp: the words of
                     // the doubles ln T and 1 / T
  i64 L2, iT2, tau2; // halves of the three (biased products)
  int rg;
  bool fast;             // T in [kTlo, kThi): fixed point
};

__device__ __forceinline__ Temp temp_of(double T, const Ctx& m, bool need_inv) {
  Temp t;
  t.T = T;
  const unsigned h = (unsigned)__double2hiint(T);
  t.fast = h - 0x40600000u < 0x40b00000u - 0x40600000u;
  int e;
  const u64 mant = mantissa(t.fast ? T : 1024.0, e);
  t.L = ((u64)e << 60) + log2_mant_q60(mant, m.rc, m.lg);
  t.iT = rcp_mant(mant, m.rc) >> (e - kTloExp);
  t.rg = T < TMID ? 0 : 1;
  const int rr = t.fast ? t.rg : 1;
  t.tau = mant >> ((rr == 0 ? kFxR0 - 1 : kFxR1 - 1) - e);
  t.L2 = (i64)(t.L >> 1); t.iT2 = (i64)(t.iT >> 1); t.tau2 = (i64)(t.tau >> 1);
  t.invT = 0.0;
  if (need_inv) t.invT = t.fast ? to_double((i64)(t.iT >> 1), 63 + kTloExp) : 1.0 / T;
  return t;
}

// ln T and 1 / T for the FP64 forms of species and reactions.  slow_temp forms them once per right-hand
// side for a temperature outside the range; the kernel of several lanes per cell, whose lanes have one
// or two species and three reactions each, forms them there.
static __device__ __noinline__ double2 ln_inv(double T) { return make_double2(log(T), 1.0 / T); }
__device__ __forceinline__ void slow_temp(Temp& t) {
  const double2 s = ln_inv(t.T);
  t.L = (u64)__double_as_longlong(s.x);
  t.iT = (u64)__double_as_longlong(s.y);
}
__device__ __forceinline__ double2 ln_inv_of(const Temp& t) {
  return t.fast ? ln_inv(t.T) : make_double2(__longlong_as_double((i64)t.L), __longlong_as_double((i64)t.iT));
}

// g/RT of species k as a double (the G array holds Q11.52 / ln 2 in fast cells, doubles in others)
__device__ __forceinline__ double g_of(double raw, bool fast) {
  return fast ? to_double(__double_as_longlong(raw), 52) * kLn2 : raw;
}

// the exponential of the FP64 forms, out of line: six copies in them cost the cells that take none of
// these forms 0.5 % (code size, presumably), and those that do 6 %
static __device__ __noinline__ double exp_slow(double x, const u64* e2) { return exp_any(x, e2); }

// Rate constants in FP64 for what the fixed-point path leaves out: cells whose temperature is
// outside its range, reactions whose exponents are.  Reaction id of the FP64 form; G: the cell's
// Gibbs energies, element k at k * stride.  kf (the high-pressure limit of a fall-off reaction),
// 1 / Kc, and k0 of a fall-off reaction; li = ln T and 1 / T.  The exponentials run on the integer pipe
// here too: 100003 H2 cells of 4100 to 5500 K take 676 ms (two lanes a cell: 745); with the library's,
// and ln T and 1 / T formed for each reaction, 1016.
static __device__ __noinline__ void slow_k(const Ctx& m, const double* G, int stride, int id, double2 li, bool fast,
                                           double* kf, double* invKc, double* k0) {
  const MechLayout& L = *m.lay;
  const double lnT = li.x, invT = li.y;
  const double* lnA = (const double*)(m.blob + L.o_lnA);
  const double* beta = (const double*)(m.blob + L.o_beta);
  const double* Ta = (const double*)(m.blob + L.o_Ta);
  const short4 re = ((const short4*)(m.blob + L.o_reac))[id], pr = ((const short4*)(m.blob + L.o_prod))[id];
  const short4 ri = ((const short4*)(m.blob + L.o_rinfo))[id];
  *kf = exp_slow(lnA[id] + beta[id] * lnT - Ta[id] * invT, m.e2);
  if (ri.x == 2) {
    const double* tr = (const double*)(m.blob + L.o_troe) + 8 * ri.w;
    *k0 = exp_slow(tr[0] + tr[1] * lnT - tr[2] * invT, m.e2);
  }
  double x = 0.0;                                   // Delta G / RT, empty slots skipped
  if (pr.x >= 0) x = g_of(G[pr.x * stride], fast);
  if (pr.y >= 0) x += g_of(G[pr.y * stride], fast);
  if (pr.z >= 0) x += g_of(G[pr.z * stride], fast);
  if (re.x >= 0) x -= g_of(G[re.x * stride], fast);
  if (re.y >= 0) x -= g_of(G[re.y * stride], fast);
  if (re.z >= 0) x -= g_of(G[re.z * stride], fast);
  if (ri.y != 0) {
    const double* cst = (const double*)(m.blob + L.o_const);
    x = fma(cst[kC_NU + 8 + ri.y], lnT - cst[kC_LNPR0], x);
  }
  *invKc = exp_slow(x, m.e2);
}

// Troe blending in FP64 from kinf, k0 and the collision-partner sum (the general form: any value
// of the arguments): kf, d ln kf/dT and d kf/d[M]
static __device__ __noinline__ void slow_troe(const Ctx& m, const FxTroe& t, double T, double invT, double kinf, double k0,
                                              double Mc, double dlnkinf, double* kf, double* dlnkf, double* dkfdM) {
  *kf = 0.0; *dlnkf = 0.0; *dkfdM = 0.0;
  if (kinf == 0.0 || k0 == 0.0) return;
  const double e3 = exp_slow(-T * t.iT3, m.e2), e1 = exp_slow(-T * t.iT1, m.e2);
  double Fc = (1.0 - t.a) * e3 + t.a * e1;
  double dFc = -(1.0 - t.a) * t.iT3 * e3 - t.a * t.iT1 * e1;
  if (t.has_t2 != 0.0) {
    const double e2 = exp_slow(-t.T2 * invT, m.e2);
    Fc += e2;
    dFc += t.T2 * invT * invT * e2;
  }
  if (Mc == 0.0) {
    *dkfdM = k0 * pow(Fc, 1.0 / (1.0 + 1.0 / (0.14 * 0.14)));
    return;
  }
  const double Prr = k0 * Mc / kinf;
  const double L = log10(Fc);
  const double n = 0.75 - 1.27 * L;
  const double u = log10(Prr) + (-0.4 - 0.67 * L);
  const double d = n - 0.14 * u;
  const double f1 = u / d;
  const double den = 1.0 + f1 * f1;
  const double F = exp_slow(2.302585092994046 * (L / den), m.e2);
  const double opr = 1.0 / (1.0 + Prr);
  *kf = kinf * (Prr * opr) * F;
  const double dGdlogPr = -2.0 * L * f1 / (den * den) * (n / (d * d));
  const double df1dL = (-0.67 * d - u * (-1.27 + 0.14 * 0.67)) / (d * d);
  const double dGdL = 1.0 / den - 2.0 * L * f1 / (den * den) * df1dL;
  const double dLdT = dFc / (Fc * 2.302585092994046);
  const double dlnPr = t.b0d * invT + t.Ta0K * invT * invT - dlnkinf;
  *dlnkf = dlnkinf + dlnPr * (opr + dGdlogPr) + 2.302585092994046 * dGdL * dLdT;
  *dkfdM = k0 * F * opr * (opr + dGdlogPr);
}

// Troe blending (Gilbert, Luther & Troe 1983): kf = kinf fac with fac = Pr / (1 + Pr) F; Xk =
// log2(k0 / kinf).  With JAC, dln receives d ln kf/dT and dM the ratio (d kf/d[M]) / kf.  False
// where a value leaves the fixed-point range (the caller then takes slow_troe).
template <bool JAC>
__device__ __forceinline__ bool troe_fast(const Ctx& m, const FxTroe& t, const Temp& q, i64 Xk, double Mc,
                                          double dlnkinf, double* fac, double* dln, double* dM) {
  constexpr double kLog10_2 = 0.30102999566398120;
  if (!exp2_in_range(Xk) || !positive_normal(Mc)) return false;
  const double e3 = exp_any(-q.T * t.iT3, m.e2), e1 = exp_any(-q.T * t.iT1, m.e2);
  double Fc = fma(t.a, e1 - e3, e3);
  double e2 = 0.0, invT = 0.0;
  if (t.has_t2 != 0.0) {
    invT = JAC ? q.invT : to_double((i64)(q.iT >> 1), 63 + kTloExp);
    e2 = exp_any(-t.T2 * invT, m.e2);
    Fc += e2;
  }
  if (!positive_normal(Fc)) return false;
  const double Prr = __dmul_rn(exp2_q52(Xk, m.e2), Mc);
  const double l2F = to_double(log2_q52(Fc, m.rc, m.lg), 52);
  // log2 k0/kinf + log2 [M] stays below 2046 in magnitude
  const double l2P = to_double(Xk + log2_q52(Mc, m.rc, m.lg), 52);
  const double L = l2F * kLog10_2;
  const double n = fma(-1.27, L, 0.75);
  const double u = fma(l2P, kLog10_2, fma(-0.67, L, -0.4));
  const double d = fma(-0.14, u, n);
  const double rd = rcp(d);
  const double f1 = u * rd;
  const double rden = rcp(fma(f1, f1, 1.0));
  const double xF = l2F * rden;
  if (!(((unsigned)__double2hiint(xF) & 0x7fffffffu) < 0x408f0000u)) return false;   // |xF| < 992
  const double F = exp2_q52(q52(xF), m.e2);
  const double opr = rcp(1.0 + Prr);
  *fac = Prr * opr * F;
  if (JAC) {
    const double g2 = -2.0 * L * f1 * rden * rden;
    const double rd2 = rd * rd;
    const double dGdlogPr = g2 * (n * rd2);
    const double df1dL = fma(-0.67, d, u * (1.27 - 0.14 * 0.67)) * rd2;
    const double dGdL = fma(g2, df1dL, rden);
    double dFc = fma(-(1.0 - t.a) * t.iT3, e3, -(t.a * t.iT1 * e1));
    if (t.has_t2 != 0.0) dFc = fma(t.T2 * invT * invT, e2, dFc);
    const double s = opr + dGdlogPr;
    const double dlnPr = fma(t.Ta0K * q.invT, q.invT, t.b0d * q.invT) - dlnkinf;
    *dln = fma(dGdL * dFc, rcp(Fc), fma(dlnPr, s, dlnkinf));
    *dM = s * rcp(Mc);
  }
  return true;
}

// Base-2 exponents of a reaction's forward and reverse rate constants: log2 kf = log2 A + b log2 T -
// Ta / (T ln 2), log2 kr = log2 kf + Delta G / (RT ln 2) - dnu log2(p_atm / (R T)); shift = iT2 - L2
// of the biased products, D = log2 T - log2(p_atm / R).
template <class R>
__device__ __forceinline__ i64 exponent_f(const R& r, const Temp& t, i64 shift) {
  return r.lnA + (i64)(umulhi3(r.beta, t.L) - umulhi3(r.Ta, t.iT)) + shift;
}

// FP64 rate constants of a reaction that (or whose cell) is outside the fixed-point range, li = ln T and
// 1 / T; kf and kr with the fall-off blending of Troe record t (nullable), d ln kf/dT, d kf/d[M] and 1 / Kc
static __device__ __noinline__ void slow_rate(const Ctx& m, const double* G, int stride, int id, const FxTroe* t, double T,
                                              double2 li, bool fast, double Mc, double* kf, double* kr, double* dlnkf,
                                              double* dkfdM, double* invKc) {
  double k0 = 0.0;
  slow_k(m, G, stride, id, li, fast, kf, invKc, &k0);
  if (t) {
    const double kinf = *kf;
    slow_troe(m, *t, T, li.y, kinf, k0, Mc, *dlnkf, kf, dlnkf, dkfdM);
  }
  *kr = *kf * *invKc;
}
static __device__ __noinline__ void slow_rate(const Ctx& m, const double* G, int stride, int id, const FxTroe* t, double T,
                                              bool fast, double Mc, double* kf, double* kr, double* dlnkf, double* dkfdM,
                                              double* invKc) {
  slow_rate(m, G, stride, id, t, T, ln_inv(T), fast, Mc, kf, kr, dlnkf, dkfdM, invKc);
}

}  // namespace fx
}  // namespace chem
