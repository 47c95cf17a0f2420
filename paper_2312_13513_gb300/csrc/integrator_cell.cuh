// Reactor right-hand side, analytic Jacobian and Rodas4 attempt of one cell in one thread, for
// small mechanisms (N = ns + 1 <= 12) with a fixed-point form (fx_mech.h).
//
// What bounds it: the FP64 pipe (fixed.cuh).  A group of two lanes per cell (integrator.cu) spends
// about 14.4 k FP64 lane slots per Rodas4 attempt of the 9-species mechanism: one lane idles
// through every per-cell scalar and through the fall-off reaction, every rate constant costs an
// FP64 exponential and its reverse a product of 1/Kc factors.  One thread per cell keeps all 32
// lanes busy, needs no group synchronisation or shuffles, reads the mechanism by warp-uniform
// addresses, and takes the rate constants of both directions straight from base-2 exponents in
// fixed point (log2 kr = log2 kf + Delta G / (RT ln 2): integer adds), so exponentials, logarithms,
// NASA-7 polynomials and reciprocals of T leave the FP64 pipe.
//
// Layout: a warp owns 32 cells; element e of a lane's workspace is at e * 32 + lane (doubles), so
// every access, also by a lane-dependent row after pivoting, is free of bank conflicts.
#pragma once

#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "chem_internal.h"
#include "fixed.cuh"
#include "queue.cuh"

namespace chem {
namespace cell {

// workspace elements of one cell (doubles): state, six stage vectors, the iteration matrix,
// concentrations, Gibbs energies and enthalpies
template <int NS>
struct Ws {
  static constexpr int N = NS + 1;
  static constexpr int Y = 0, U = N, M = 7 * N, C = M + N * N, G = C + NS, H = G + NS, TOTAL = H + NS;
  // scratch inside the stage vectors while the Jacobian is formed (u_0 holds the rates)
  static constexpr int DWDT = U + N, CP = U + 2 * N, RK = U + 3 * N, HM = U + 4 * N;
};

struct View {
  const fx::u64 *e2, *lg;
  const uint32_t* rc;
  const FxSpecies* sp;
  const double *W, *invW, *nu, *effv, *eff;
  const FxReac* reac;
  const FxTroe* troe;
  const int16_t* effidx;
  const int* effoff;
  int nr;
  fx::i64 lpr0;
  const unsigned char* blob;     // FP64 form in global memory (rates outside the fixed-point range)
  const MechLayout* lay;
};

__device__ __forceinline__ View bind(const unsigned char* s, const FxLayout& L, const unsigned char* blob,
                                     const MechLayout* lay) {
  View v;
  v.e2 = (const fx::u64*)(s + L.o_exp2);
  v.lg = (const fx::u64*)(s + L.o_lg);
  v.rc = (const uint32_t*)(s + L.o_rcp);
  v.sp = (const FxSpecies*)(s + L.o_sp);
  v.W = (const double*)(s + L.o_W);
  v.invW = (const double*)(s + L.o_invW);
  v.nu = (const double*)(s + L.o_nu);
  v.effv = (const double*)(s + L.o_effv);
  v.eff = (const double*)(s + L.o_eff);
  v.reac = (const FxReac*)(s + L.o_reac);
  v.troe = (const FxTroe*)(s + L.o_troe);
  v.effidx = (const int16_t*)(s + L.o_effidx);
  v.effoff = (const int*)(s + L.o_effoff);
  v.nr = L.nr;
  v.lpr0 = L.lpr0;
  v.blob = blob;
  v.lay = lay;
  return v;
}

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
__device__ __forceinline__ double exp_any(double x, const fx::u64* e2) {
  const unsigned hx = (unsigned)__double2hiint(x) & 0x7fffffffu;
  if (hx >= 0x4085e000u) return (__double2hiint(x) < 0 && hx < 0x7ff00000u && hx >= 0x40900000u) ? 0.0 : exp(x);
  // x log2 e: |x| < 1024 in Q10.53 times log2 e in Q1.63, a Q11.52 product
  const fx::i64 q = fx::q52(x) * 2;
  return fx::exp2_q52(fx::mulhi_su(q, fx::kLog2e), e2);
}

// log2 x as Q11.52 in range only: x positive, normal, finite (the caller's test)
__device__ __forceinline__ bool positive_normal(double x) {
  return (unsigned)__double2hiint(x) - 0x00100000u < 0x7ff00000u - 0x00100000u;
}

// thermo state of a right-hand side at one temperature
struct Temp {
  double T, invT;
  fx::u64 L, iT, tau;    // log2 T (Q4.60), 128 / T and T / 2^r (Q0.64)
  int rg;
  bool fast;             // T in [kTlo, kThi): fixed point
};

__device__ __forceinline__ Temp temp_of(double T, const View& m, bool need_inv) {
  Temp t;
  t.T = T;
  const unsigned h = (unsigned)__double2hiint(T);
  t.fast = h - 0x40600000u < 0x40b00000u - 0x40600000u;
  int e;
  const fx::u64 mant = fx::mantissa(t.fast ? T : 1024.0, e);
  t.L = ((fx::u64)e << 60) + fx::log2_mant_q60(mant, m.rc, m.lg);
  t.iT = fx::rcp_mant(mant, m.rc) >> (e - fx::kTloExp);
  t.rg = T < TMID ? 0 : 1;
  const int rr = t.fast ? t.rg : 1;
  t.tau = mant >> ((rr == 0 ? kFxR0 - 1 : kFxR1 - 1) - e);
  t.invT = 0.0;
  if (need_inv) t.invT = t.fast ? fx::to_double((fx::i64)(t.iT >> 1), 63 + fx::kTloExp) : 1.0 / T;
  return t;
}

// g/RT of species k as a double (the G array holds Q11.52 / ln 2 in fast cells, doubles in others)
__device__ __forceinline__ double g_of(double raw, bool fast) {
  return fast ? fx::to_double(__double_as_longlong(raw), 52) * fx::kLn2 : raw;
}

// Rate constants in FP64 for what the fixed-point path leaves out: cells whose temperature is
// outside its range, reactions whose exponents are.  kf (the high-pressure limit of a fall-off
// reaction) and 1 / Kc; k0 of a fall-off reaction.
template <int NS>
__device__ __noinline__ void slow_k(const View& m, const double* col, int j, double T, bool fast, double* kf,
                                    double* invKc, double* k0) {
  using w = Ws<NS>;
  const FxReac& R = m.reac[j];
  const MechLayout& L = *m.lay;
  const double lnT = log(T), invT = 1.0 / T;
  const double* lnA = (const double*)(m.blob + L.o_lnA);
  *kf = exp(lnA[j] + R.b * lnT - R.TaK * invT);
  if (R.type == 2) {
    const double* tr = (const double*)(m.blob + L.o_troe) + 8 * R.troe;
    *k0 = exp(tr[0] + tr[1] * lnT - tr[2] * invT);
  }
  double dG = 0.0;
  for (int i = 0; i < R.nre; ++i) dG -= g_of(col[(w::G + R.re[i]) * 32], fast);
  for (int i = 0; i < R.npr; ++i) dG += g_of(col[(w::G + R.pr[i]) * 32], fast);
  const double* cst = (const double*)(m.blob + L.o_const);
  *invKc = exp(dG - (double)R.dnu * (cst[kC_LNPR0] - lnT));
}

// Species thermo in FP64 (temperatures outside the fixed-point range): g/RT and h/RT (cp/R with
// jac) into the workspace; sum c cp/R and its temperature derivative, c = Y / W in the workspace
template <int NS>
__device__ __noinline__ void slow_species(const View& m, double* col, double T, double* cp_out, double* dcp_out,
                                          bool jac) {
  using w = Ws<NS>;
  const MechLayout& L = *m.lay;
  const int rg = T < TMID ? 0 : 1;
  const double lnT = log(T), invT = 1.0 / T;
  double cps = 0.0, dcps = 0.0;
  for (int k = 0; k < NS; ++k) {
    const double* hc = (const double*)(m.blob + L.o_hc) + (rg * NS + k) * 6;
    const double* sc = (const double*)(m.blob + L.o_sc) + (rg * NS + k) * 6;
    const double* cc = (const double*)(m.blob + L.o_cpc) + (rg * NS + k) * 5;
    const double h = hc[0] + T * (hc[1] + T * (hc[2] + T * (hc[3] + T * hc[4]))) + hc[5] * invT;
    const double s = sc[0] * lnT + T * (sc[1] + T * (sc[2] + T * (sc[3] + T * sc[4]))) + sc[5];
    const double cp = cc[0] + T * (cc[1] + T * (cc[2] + T * (cc[3] + T * cc[4])));
    col[(w::G + k) * 32] = h - s;
    col[(w::H + k) * 32] = h;
    const double c = col[(w::C + k) * 32];
    cps = fma(c, cp, cps);
    if (jac) {
      dcps += c * (cc[1] + T * (2.0 * cc[2] + T * (3.0 * cc[3] + T * (4.0 * cc[4]))));
      col[(w::CP + k) * 32] = cp;
    }
  }
  *cp_out = cps;
  *dcp_out = dcps;
}

// Troe blending in FP64 from kinf, k0 and the collision-partner sum (the general form: any value
// of the arguments): kf, d ln kf/dT and d kf/d[M]
__device__ __noinline__ void slow_troe(const FxTroe& t, double T, double kinf, double k0, double Mc, double dlnkinf,
                                       double* kf, double* dlnkf, double* dkfdM) {
  const double invT = 1.0 / T;
  *kf = 0.0; *dlnkf = 0.0; *dkfdM = 0.0;
  if (kinf == 0.0 || k0 == 0.0) return;
  const double e3 = exp(-T * t.iT3), e1 = exp(-T * t.iT1);
  double Fc = (1.0 - t.a) * e3 + t.a * e1;
  double dFc = -(1.0 - t.a) * t.iT3 * e3 - t.a * t.iT1 * e1;
  if (t.has_t2 != 0.0) {
    const double e2 = exp(-t.T2 * invT);
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
  const double F = exp(2.302585092994046 * (L / den));
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
__device__ __forceinline__ bool troe_fast(const View& m, const FxTroe& t, const Temp& q, fx::i64 Xk, double Mc,
                                          double dlnkinf, double* fac, double* dln, double* dM) {
  constexpr double kLog10_2 = 0.30102999566398120;
  if (!fx::exp2_in_range(Xk) || !positive_normal(Mc)) return false;
  const double e3 = exp_any(-q.T * t.iT3, m.e2), e1 = exp_any(-q.T * t.iT1, m.e2);
  double Fc = fma(t.a, e1 - e3, e3);
  double e2 = 0.0, invT = 0.0;
  if (t.has_t2 != 0.0) {
    invT = JAC ? q.invT : fx::to_double((fx::i64)(q.iT >> 1), 63 + fx::kTloExp);
    e2 = exp_any(-t.T2 * invT, m.e2);
    Fc += e2;
  }
  if (!positive_normal(Fc)) return false;
  const double Prr = fx::exp2_q52(Xk, m.e2) * Mc;
  const double l2F = fx::to_double(fx::log2_q52(Fc, m.rc, m.lg), 52);
  // log2 k0/kinf + log2 [M] stays below 2046 in magnitude
  const double l2P = fx::to_double(Xk + fx::log2_q52(Mc, m.rc, m.lg), 52);
  const double L = l2F * kLog10_2;
  const double n = fma(-1.27, L, 0.75);
  const double u = fma(l2P, kLog10_2, fma(-0.67, L, -0.4));
  const double d = fma(-0.14, u, n);
  const double rd = rcp(d);
  const double f1 = u * rd;
  const double rden = rcp(fma(f1, f1, 1.0));
  const double xF = l2F * rden;
  if (!(((unsigned)__double2hiint(xF) & 0x7fffffffu) < 0x408f0000u)) return false;   // |xF| < 992
  const double F = fx::exp2_q52(fx::q52(xF), m.e2);
  const double opr = rcp(1.0 + Prr);
  *fac = Prr * opr * F;
  if (JAC) {
    const double g2 = -2.0 * L * f1 * rden * rden;
    const double rd2 = rd * rd;
    const double dGdlogPr = g2 * (n * rd2);
    const double df1dL = fma(-0.67, d, u * (1.27 - 0.14 * 0.67)) * rd2;
    const double dGdL = fma(g2, df1dL, rden);
    double dFc = -(1.0 - t.a) * t.iT3 * e3 - t.a * t.iT1 * e1;
    if (t.has_t2 != 0.0) dFc += t.T2 * invT * invT * e2;
    const double s = opr + dGdlogPr;
    const double dlnPr = fma(t.Ta0K * q.invT, q.invT, t.b0d * q.invT) - dlnkinf;
    *dln = dlnkinf + dlnPr * s + dGdL * dFc * rcp(Fc);
    *dM = s * rcp(Mc);
  }
  return true;
}

// Right-hand side f(T, Y) into u (workspace elements uoff ..), and with JAC the NEGATED analytic
// Jacobian -df/dy into the matrix.  Yk(k) returns the mass fraction of species k; p and 1 / p of
// the cell.  Writes the concentrations, Gibbs energies and enthalpies of the workspace.
template <int NS, bool JAC, class YF>
__device__ __forceinline__ void rhs(const View& m, double* col, double T, YF Yk, double p, double invp, int uoff) {
  using w = Ws<NS>;
  constexpr int N = w::N;
  const Temp t = temp_of(T, m, JAC);
  double S = 0.0, cps = 0.0, dcps = 0.0;
  double c[NS];
#pragma unroll
  for (int k = 0; k < NS; ++k) {
    c[k] = Yk(k) * m.invW[k];
    S += c[k];
    col[(w::C + k) * 32] = c[k];
  }
  if (t.fast) {
    const FxSpecies* sp = m.sp + t.rg * NS;
#pragma unroll 3
    for (int k = 0; k < NS; ++k) {
      const FxSpecies& s = sp[k];
      fx::i64 g = s.g[4], h = s.h[4], cp = s.c[4];
#pragma unroll
      for (int i = 3; i >= 0; --i) {
        g = fx::mulhi_su(g, t.tau) + s.g[i];
        h = fx::mulhi_su(h, t.tau) + s.h[i];
        cp = fx::mulhi_su(cp, t.tau) + s.c[i];
      }
      g += fx::mulhi_su(s.ga6, t.iT) + fx::mulhi_su(s.gl, t.L);
      h += fx::mulhi_su(s.ha6, t.iT);
      col[(w::G + k) * 32] = __longlong_as_double(g);
      col[(w::H + k) * 32] = fx::to_double(h, 52);
      const double cpd = fx::to_double(cp, 52);
      const double ck = col[(w::C + k) * 32];
      cps = fma(ck, cpd, cps);
      if (JAC) {
        // d(cp/R)/dT 2^r = sum_i i c_i tau^(i-1)
        fx::i64 dc = s.c[4] * 4;
        dc = fx::mulhi_su(dc, t.tau) + s.c[3] * 3;
        dc = fx::mulhi_su(dc, t.tau) + s.c[2] * 2;
        dc = fx::mulhi_su(dc, t.tau) + s.c[1];
        dcps = fma(ck, fx::to_double(dc, 52 + (t.rg == 0 ? kFxR0 : kFxR1)), dcps);
        col[(w::CP + k) * 32] = cpd;
      }
    }
  } else {
    slow_species<NS>(m, col, T, &cps, &dcps, JAC);
  }
  const double RTS = RU * T * S;
  const double rho = p * rcp(RTS), invrho = RTS * invp;
#pragma unroll
  for (int k = 0; k < NS; ++k) {
    col[(w::C + k) * 32] = rho * c[k];
    col[(uoff + 1 + k) * 32] = 0.0;
    if (JAC) col[(w::DWDT + k) * 32] = 0.0;
  }
  if (JAC) {
#pragma unroll
    for (int e = 0; e < NS * NS; ++e) col[(w::M + (1 + e / NS) * N + 1 + e % NS) * 32] = 0.0;
  }
  const double Ctot = rho * S;
  const fx::i64 L52 = (fx::i64)((t.L + 128ull) >> 8);
  double* Jm = col + (w::M + N + 1) * 32;      // row 1 (species 0), column 1

  for (int j = 0; j < m.nr; ++j) {
    const FxReac& R = m.reac[j];
    const int nre = R.nre, npr = R.npr;
    const fx::i64 Xf = R.lnA + fx::mulhi_su(R.beta, t.L) - fx::mulhi_su(R.Ta, t.iT);
    const double* cr0 = col + (w::C + R.re[0]) * 32;
    const double* cp0 = col + (w::C + R.pr[0]) * 32;
    double a0 = cr0[0], b0 = cp0[0], a1 = 1.0, a2 = 1.0, b1 = 1.0, b2 = 1.0;
    fx::i64 Xr = Xf + __double_as_longlong(cp0[NS * 32]) - __double_as_longlong(cr0[NS * 32]);   // G follows C
    double Pf = a0, Pr = b0;
    if (nre > 1) {
      const double* q = col + (w::C + R.re[1]) * 32;
      a1 = q[0]; Xr -= __double_as_longlong(q[NS * 32]); Pf *= a1;
      if (nre > 2) {
        const double* q2 = col + (w::C + R.re[2]) * 32;
        a2 = q2[0]; Xr -= __double_as_longlong(q2[NS * 32]); Pf *= a2;
      }
    }
    if (npr > 1) {
      const double* q = col + (w::C + R.pr[1]) * 32;
      b1 = q[0]; Xr += __double_as_longlong(q[NS * 32]); Pr *= b1;
      if (npr > 2) {
        const double* q2 = col + (w::C + R.pr[2]) * 32;
        b2 = q2[0]; Xr += __double_as_longlong(q2[NS * 32]); Pr *= b2;
      }
    }
    const int dnu = R.dnu;
    Xr += (fx::i64)dnu * (L52 - m.lpr0);
    double Mc = 1.0;
    if (R.type != 0) {
      Mc = Ctot;
      const int e1 = m.effoff[R.tb + 1];
      for (int e = m.effoff[R.tb]; e < e1; ++e) Mc = fma(m.effv[e], col[(w::C + m.effidx[e]) * 32], Mc);
    }
    double dlnkf = 0.0;
    if (JAC) dlnkf = fma(R.TaK * t.invT, t.invT, R.b * t.invT);
    double kf, kr, k0 = 0.0, dMr = 0.0;        // dMr: (d kf / d[M]) / kf of a fall-off reaction
    double dkfdM = 0.0, invKc = 0.0;
    bool done = t.fast && !R.slow && fx::exp2_in_range(Xf) && fx::exp2_in_range(Xr);
    if (done) {
      kf = fx::exp2_q52(Xf, m.e2);
      kr = fx::exp2_q52(Xr, m.e2);
      if (R.type == 2) {
        const FxTroe& F = m.troe[R.troe];
        const fx::i64 Xk = F.lnA0 + fx::mulhi_su(F.b0, t.L) - fx::mulhi_su(F.Ta0, t.iT) - Xf;
        double fac = 1.0, dl = 0.0;
        done = troe_fast<JAC>(m, F, t, Xk, Mc, dlnkf, &fac, &dl, &dMr);
        kf *= fac;
        kr *= fac;
        if (JAC && done) dlnkf = dl;
      }
    }
    const bool fastk = done;
    if (!fastk) {
      slow_k<NS>(m, col, j, T, t.fast, &kf, &invKc, &k0);
      if (R.type == 2) {
        const double kinf = kf;
        double dl;
        slow_troe(m.troe[R.troe], T, kinf, k0, Mc, dlnkf, &kf, &dl, &dkfdM);
        dlnkf = dl;
      }
      kr = kf * invKc;
    }
    double* wd = col + (uoff + 1) * 32;
    if (!JAC) {
      double q = fma(kf, Pf, -(kr * Pr));
      if (R.type == 1) q *= Mc;
      const int nn = R.nnet;
      for (int i = 0; i < nn; ++i) {
        double* x = wd + R.sp[i] * 32;
        *x = fma(m.nu[R.nu[i] + 8], q, *x);
      }
    } else {
      const double fwd = kf * Pf, rev = kr * Pr, net = fwd - rev;
      const double mult = R.type == 1 ? Mc : 1.0;
      double dH = -(double)dnu;
      for (int i = 0; i < nre; ++i) dH -= col[(w::H + R.re[i]) * 32];
      for (int i = 0; i < npr; ++i) dH += col[(w::H + R.pr[i]) * 32];
      const double dlnKc = dH * t.invT;
      double dqdT = fma(net, dlnkf, rev * dlnKc);
      double q = net, ka = kf, kb = kr;
      if (R.type == 1) { q *= mult; dqdT *= mult; ka *= mult; kb *= mult; }
      const int nn = R.nnet;
      for (int i = 0; i < nn; ++i) {
        const double nu = m.nu[R.nu[i] + 8];
        double* x = wd + R.sp[i] * 32;
        *x = fma(nu, q, *x);
        double* y = col + (w::DWDT + R.sp[i]) * 32;
        *y = fma(nu, dqdT, *y);
      }
      // d(wdot)/dC, negated: a slot's derivative times the net coefficient of every species
      auto slot = [&](int sp, double d) {
        for (int i = 0; i < nn; ++i) {
          double* x = Jm + (R.sp[i] * N + sp) * 32;
          *x = fma(-m.nu[R.nu[i] + 8], d, *x);
        }
      };
      if (nre == 1) {
        slot(R.re[0], ka);
      } else if (nre == 2) {
        slot(R.re[0], ka * a1);
        slot(R.re[1], ka * a0);
      } else {
        slot(R.re[0], ka * a1 * a2);
        slot(R.re[1], ka * a0 * a2);
        slot(R.re[2], ka * a0 * a1);
      }
      if (npr == 1) {
        slot(R.pr[0], -kb);
      } else if (npr == 2) {
        slot(R.pr[0], -kb * b1);
        slot(R.pr[1], -kb * b0);
      } else {
        slot(R.pr[0], -kb * b1 * b2);
        slot(R.pr[1], -kb * b0 * b2);
        slot(R.pr[2], -kb * b0 * b1);
      }
      if (R.type != 0) {
        double X;
        if (R.type == 1) X = net;
        else X = fastk ? dMr * net : dkfdM * (Pf - Pr * invKc);
        const double* ef = m.eff + R.tb * NS;
        for (int i = 0; i < nn; ++i) {
          const double nx = -m.nu[R.nu[i] + 8] * X;
          double* x = Jm + R.sp[i] * N * 32;
#pragma unroll
          for (int mm = 0; mm < NS; ++mm) x[mm * 32] = fma(nx, ef[mm], x[mm * 32]);
        }
      }
    }
  }

  // species and temperature rows: f_k = W_k w_k / rho, f_0 = -T sum h/RT w / (rho cp/R)
  double Q = 0.0, r31 = 0.0, r32 = 0.0;
  double wk[NS];
#pragma unroll
  for (int k = 0; k < NS; ++k) {
    wk[k] = col[(uoff + 1 + k) * 32];
    const double h = col[(w::H + k) * 32];
    Q = fma(h, wk[k], Q);
    if (JAC) {
      r31 = fma(col[(w::CP + k) * 32], wk[k], r31);
      r32 = fma(h, col[(w::DWDT + k) * 32], r32);
    }
    col[(uoff + 1 + k) * 32] = m.W[k] * (wk[k] * invrho);
  }
  const double ircp = rcp(rho * cps);         // 1 / (rho cp/R)
  col[uoff * 32] = -(T * Q) * ircp;
  if (!JAC) return;

  // chain rule through C(T, Y) and rho(T, Y), as in integrator.cu with cp and h in units of R:
  //   J_km = W_k / W_m (dw_k/dC_m - (r_k - w_k) rho^-1 / S), J_k0 = W_k / rho (dw_k/dT - (r_k - w_k) / T)
  //   J_0m = (-(rho H_m - R_h / S) + Q' rho (cp_m - cp / S)) / (rho cp W_m), Q' = Q / (rho cp)
  const double iS = rcp(S);
  const double rS = invrho * iS;
  double Rh = 0.0;
#pragma unroll
  for (int k = 0; k < NS; ++k) {
    double s = 0.0;
#pragma unroll
    for (int mm = 0; mm < NS; ++mm) s = fma(Jm[(k * N + mm) * 32], col[(w::C + mm) * 32], s);
    Rh = fma(-col[(w::H + k) * 32], s, Rh);
    const double dk = -s - wk[k];
    col[(w::RK + k) * 32] = dk * rS;
    Jm[(k * N - 1) * 32] = -(m.W[k] * invrho * (col[(w::DWDT + k) * 32] - dk * t.invT));
  }
  const double TQ = T * Q, TRh = T * Rh;
  const double Qr = TQ * ircp;                 // -f_0
  col[w::M * 32] = (r31 + T * r32 - Rh) * ircp + Qr * (cps * t.invT - dcps) * (rho * ircp);
  const double RhS = TRh * iS, cpS = cps * iS, Qrr = Qr * rho;
#pragma unroll
  for (int mm = 0; mm < NS; ++mm) {
    double s = 0.0;
#pragma unroll
    for (int k = 0; k < NS; ++k) s = fma(-col[(w::H + k) * 32], Jm[(k * N + mm) * 32], s);
    const double Hm = T * s;
    Jm[(mm - N) * 32] = m.invW[mm] * ircp * ((rho * Hm - RhS) - Qrr * (col[(w::CP + mm) * 32] - cpS));
  }
#pragma unroll
  for (int k = 0; k < NS; ++k) {
    const double rk = col[(w::RK + k) * 32], Wk = m.W[k];
#pragma unroll
    for (int mm = 0; mm < NS; ++mm) {
      double* x = Jm + (k * N + mm) * 32;
      *x = Wk * m.invW[mm] * (rk + *x);
    }
  }
}

}  // namespace cell
}  // namespace chem
