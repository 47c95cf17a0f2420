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
// NASA-7 polynomials and reciprocals of T leave the FP64 pipe: about 4.5 k FP64 instructions per
// attempt of 32 cells instead of 14.4 k of 16; 2^20 flame cells 242 -> 108 ms (80 with eight warps
// an SM, integrator_cell.cu).
//
// Sums that a compiler could contract in more than one way are written as explicit FMAs: the kernel
// for few cells (integrator_coop.cu) does the same operations in the same order, so that a cell's
// result does not depend on the launch it is part of.
//
// Layout: a warp owns 32 cells; element e of a lane's workspace is at e * 32 + lane (doubles), so
// every access, also by a lane-dependent row after pivoting, is free of bank conflicts.  The matrix
// is a second array of the same form: in shared memory, or for large launches in global memory
// (integrator_cell.cu).
#pragma once

#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include "chem_internal.h"
#include "fx_rates.cuh"
#include "queue.cuh"

namespace chem {
namespace cell {

using fx::exponent_f;
using fx::rcp;
using fx::slow_temp;
using fx::Temp;
using fx::temp_of;
using fx::troe_fast;

// workspace elements of one cell (doubles): state, six stage vectors, concentrations and Gibbs
// energies (each with the empty slot's 1 and 0 at the end), enthalpies: VEC of them, and the
// iteration matrix
template <int NS>
struct Ws {
  static constexpr int N = NS + 1;
  static constexpr int Y = 0, U = N, C = 7 * N, G = C + N, H = G + N, VEC = H + NS, TOTAL = VEC + N * N;
  // scratch inside the stage vectors while the Jacobian is formed (u_0 holds the rates)
  static constexpr int DWDT = U + N, CP = U + 2 * N, RK = U + 3 * N, WK = U + 4 * N;
};

struct View : fx::Ctx {
  const FxSpecies* sp;
  const double *W, *invW, *nu, *effv, *eff;
  const FxRate* rate;
  const FxReac* reac;
  const FxTroe* troe;
  const int16_t* effidx;
  const int* effoff;
  int n_plain, n_tb, n_fo, n_gen;
  fx::i64 lpr0;
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
  v.rate = (const FxRate*)(s + L.o_rate);
  v.reac = (const FxReac*)(s + L.o_reac);
  v.troe = (const FxTroe*)(s + L.o_troe);
  v.effidx = (const int16_t*)(s + L.o_effidx);
  v.effoff = (const int*)(s + L.o_effoff);
  v.n_plain = L.n_plain; v.n_tb = L.n_tb; v.n_fo = L.n_fo; v.n_gen = L.n_gen;
  v.lpr0 = L.lpr0;
  v.blob = blob;
  v.lay = lay;
  return v;
}

// Species k in FP64 (temperatures outside the fixed-point range): g/RT, h/RT, cp/R, d(cp/R)/dT
struct Species64 {
  double g, h, cp, dcp;
};
static __device__ __noinline__ Species64 species64(const View& m, int ns, int k, double T, double2 li) {
  const MechLayout& L = *m.lay;
  const int rg = T < TMID ? 0 : 1;
  const double lnT = li.x, invT = li.y;
  const double* hc = (const double*)(m.blob + L.o_hc) + (rg * ns + k) * 6;
  const double* sc = (const double*)(m.blob + L.o_sc) + (rg * ns + k) * 6;
  const double* cc = (const double*)(m.blob + L.o_cpc) + (rg * ns + k) * 5;
  Species64 r;
  r.h = hc[0] + T * (hc[1] + T * (hc[2] + T * (hc[3] + T * hc[4]))) + hc[5] * invT;
  r.g = r.h - (sc[0] * lnT + T * (sc[1] + T * (sc[2] + T * (sc[3] + T * sc[4]))) + sc[5]);
  r.cp = cc[0] + T * (cc[1] + T * (cc[2] + T * (cc[3] + T * cc[4])));
  r.dcp = cc[1] + T * (2.0 * cc[2] + T * (3.0 * cc[3] + T * (4.0 * cc[4])));
  return r;
}
static __device__ __noinline__ Species64 species64(const View& m, int ns, int k, double T) {
  return species64(m, ns, k, T, fx::ln_inv(T));
}
// all species of a cell into its workspace (cp/R with jac); sum c cp/R and its temperature
// derivative, c = Y / W in the workspace
template <int NS>
__device__ __noinline__ void slow_species(const View& m, double* col, double T, double2 li, double* cp_out, double* dcp_out,
                                          bool jac) {
  using w = Ws<NS>;
  double cps = 0.0, dcps = 0.0;
  for (int k = 0; k < NS; ++k) {
    const Species64 r = species64(m, NS, k, T, li);
    col[(w::G + k) * 32] = r.g;
    col[(w::H + k) * 32] = r.h;
    const double c = col[(w::C + k) * 32];
    cps = fma(c, r.cp, cps);
    if (jac) {
      dcps = fma(c, r.dcp, dcps);
      col[(w::CP + k) * 32] = r.cp;
    }
  }
  *cp_out = cps;
  *dcp_out = dcps;
}

// The slots of an FxRate, warp-uniform, in registers
struct Slots {
  unsigned r0, r1, p0, p1;
};
__device__ __forceinline__ Slots slots(const uint16_t* c) {
  const uint2 v = *reinterpret_cast<const uint2*>(c);
  return Slots{v.x & 0xffffu, v.x >> 16, v.y & 0xffffu, v.y >> 16};
}
__device__ __forceinline__ double* at(double* col, unsigned off) {
  return reinterpret_cast<double*>(reinterpret_cast<unsigned char*>(col) + off);
}

// collision-partner concentration sum_k eff_k C_k of third-body set tb
template <int NS>
__device__ __forceinline__ double partners(const View& m, const double* col, int tb, double Ctot) {
  double Mc = Ctot;
  const int e1 = m.effoff[tb + 1];
  for (int e = m.effoff[tb]; e < e1; ++e) Mc = fma(m.effv[e], col[(Ws<NS>::C + m.effidx[e]) * 32], Mc);
  return Mc;
}

// Any reaction (FxReac): three species on a side, up to six net species.  Adds its production rates
// and, with JAC, its derivatives.
template <int NS, bool JAC>
__device__ __noinline__ void general_reaction(const View& m, double* col, double* Mx, const FxReac& R, const Temp& t, double T,
                                              fx::i64 shift, fx::i64 D, double Ctot, int uoff) {
  using w = Ws<NS>;
  constexpr int N = w::N;
  const int nre = R.nre, npr = R.npr, nn = R.nnet;
  const double* Cc = col + w::C * 32;
  const double* Gc = col + w::G * 32;
  const fx::i64 Xf = exponent_f(R, t, shift);
  fx::i64 Xr = Xf + (fx::i64)R.dnu * D;
  double a[3] = {1.0, 1.0, 1.0}, b[3] = {1.0, 1.0, 1.0};
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    if (i < nre) { a[i] = Cc[R.re[i] * 32]; Xr -= __double_as_longlong(Gc[R.re[i] * 32]); }
    if (i < npr) { b[i] = Cc[R.pr[i] * 32]; Xr += __double_as_longlong(Gc[R.pr[i] * 32]); }
  }
  const double Mc = R.type != 0 ? partners<NS>(m, col, R.tb, Ctot) : 1.0;
  double dlnkf = JAC ? fma(R.TaK * t.invT, t.invT, R.b * t.invT) : 0.0;
  double kf = 0.0, kr = 0.0, dMr = 0.0, dkfdM = 0.0, invKc = 0.0;
  bool fastk = t.fast && fx::exp2_in_range(Xf) && fx::exp2_in_range(Xr);
  if (fastk) {
    kf = fx::exp2_q52(Xf, m.e2);
    kr = fx::exp2_q52(Xr, m.e2);
    if (R.type == 2) {
      const FxTroe& F = m.troe[R.troe];
      const fx::i64 Xk = F.lnA0 + (fx::i64)(fx::umulhi3(F.b0, t.L) - fx::umulhi3(F.Ta0, t.iT)) + shift - Xf;
      double fac = 1.0, dl = 0.0;
      fastk = troe_fast<JAC>(m, F, t, Xk, Mc, dlnkf, &fac, &dl, &dMr);
      kf *= fac;
      kr *= fac;
      if (JAC && fastk) dlnkf = dl;
    }
  }
  if (!fastk)
    fx::slow_rate(m, Gc, 32, R.id, R.type == 2 ? m.troe + R.troe : nullptr, T, fx::ln_inv_of(t), t.fast,
                  Mc, &kf, &kr, &dlnkf, &dkfdM, &invKc);
  const double Pf = a[0] * a[1] * a[2], Pr = b[0] * b[1] * b[2];
  const double mult = R.type == 1 ? Mc : 1.0;
  const double fwd = kf * Pf, rev = kr * Pr, net = fwd - rev;
  double dqdT = 0.0;
  if (JAC) {
    double dH = -(double)R.dnu;
    for (int i = 0; i < nre; ++i) dH -= col[(w::H + R.re[i]) * 32];
    for (int i = 0; i < npr; ++i) dH += col[(w::H + R.pr[i]) * 32];
    dqdT = mult * fma(net, dlnkf, rev * (dH * t.invT));
  }
  double* Jm = Mx + (N + 1) * 32;
  for (int i = 0; i < nn; ++i) {
    const double nu = m.nu[R.nu[i] + 8];
    double* x = col + (uoff + 1 + R.sp[i]) * 32;
    *x = fma(nu, mult * net, *x);
    if (!JAC) continue;
    double* y = col + (w::DWDT + R.sp[i]) * 32;
    *y = fma(nu, dqdT, *y);
    double* row = Jm + R.sp[i] * N * 32;
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      if (q < nre) row[R.re[q] * 32] = fma(-nu, mult * kf * a[(q + 1) % 3] * a[(q + 2) % 3], row[R.re[q] * 32]);
      if (q < npr) row[R.pr[q] * 32] = fma(nu, mult * kr * b[(q + 1) % 3] * b[(q + 2) % 3], row[R.pr[q] * 32]);
    }
    if (R.type != 0) {
      const double X = R.type == 1 ? net : (fastk ? dMr * net : dkfdM * (Pf - Pr * invKc));
      const double* ef = m.eff + R.tb * NS;
      for (int mm = 0; mm < NS; ++mm) row[mm * 32] = fma(-nu * X, ef[mm], row[mm * 32]);
    }
  }
}

// Right-hand side f(T, Y) into workspace elements uoff .., and with JAC the NEGATED analytic
// Jacobian -df/dy into the matrix Mx.  Yk(k) returns the mass fraction of species k; p and 1 / p of
// the cell.  Writes the concentrations, Gibbs energies and enthalpies of the workspace.
template <int NS, bool JAC, class YF>
__device__ __forceinline__ void rhs(const View& m, double* col, double* Mx, double T, YF Yk, double p, double invp, int uoff) {
  using w = Ws<NS>;
  constexpr int N = w::N;
  Temp t = temp_of(T, m, JAC);
  double S = 0.0, cps = 0.0, dcps = 0.0;
  double c[NS];
#pragma unroll
  for (int k = 0; k < NS; ++k) {
    c[k] = __dmul_rn(Yk(k), m.invW[k]);
    S += c[k];
    col[(w::C + k) * 32] = c[k];
  }
  if (t.fast) {
    const FxSpecies* sp = m.sp + t.rg * NS;
    const fx::u64 B = 0x8000000000000000ull;
    const fx::i64 gT = t.iT2 + t.L2;
#pragma unroll 3
    for (int k = 0; k < NS; ++k) {
      const FxSpecies& s = sp[k];
      fx::u64 g = (fx::u64)s.g[4], h = (fx::u64)s.h[4], cp = (fx::u64)s.c[4];   // biased
#pragma unroll
      for (int i = 3; i >= 0; --i) {
        const fx::u64 b = i ? B : 0ull;                                        // the last one unbiased
        g = (fx::umulhi3(g, t.tau) + (fx::u64)(s.g[i] - t.tau2)) ^ b;
        h = (fx::umulhi3(h, t.tau) + (fx::u64)(s.h[i] - t.tau2)) ^ b;
        cp = (fx::umulhi3(cp, t.tau) + (fx::u64)(s.c[i] - t.tau2)) ^ b;
      }
      g += fx::umulhi3((fx::u64)s.ga6, t.iT) + fx::umulhi3((fx::u64)s.gl, t.L) - (fx::u64)gT;
      h += fx::umulhi3((fx::u64)s.ha6, t.iT) - (fx::u64)t.iT2;
      col[(w::G + k) * 32] = __longlong_as_double((fx::i64)g);
      col[(w::H + k) * 32] = fx::to_double((fx::i64)h, 52);
      const double cpd = fx::to_double((fx::i64)cp, 52);
      const double ck = col[(w::C + k) * 32];
      cps = fma(ck, cpd, cps);
      if (JAC) {
        // d(cp/R)/dT 2^r = sum_i i c_i tau^(i-1)
        fx::u64 dc = fx::biased((fx::i64)(((fx::u64)s.c[4] ^ B) << 2));
        dc = (fx::umulhi3(dc, t.tau) + (fx::u64)(s.c[3] * 3 - t.tau2)) ^ B;
        dc = (fx::umulhi3(dc, t.tau) + (fx::u64)(s.c[2] * 2 - t.tau2)) ^ B;
        dc = fx::umulhi3(dc, t.tau) + (fx::u64)(s.c[1] - t.tau2);
        dcps = fma(ck, fx::to_double((fx::i64)dc, 52 + (t.rg == 0 ? kFxR0 : kFxR1)), dcps);
        col[(w::CP + k) * 32] = cpd;
      }
    }
  } else {
    slow_temp(t);
    slow_species<NS>(m, col, T, fx::ln_inv_of(t), &cps, &dcps, JAC);
  }
  const double RTS = RU * T * S;
  const double rho = p * rcp(RTS), invrho = RTS * invp;
#pragma unroll
  for (int k = 0; k < NS; ++k) {
    col[(w::C + k) * 32] = rho * c[k];
    col[(uoff + 1 + k) * 32] = 0.0;
    if (JAC) col[(w::DWDT + k) * 32] = 0.0;
  }
  col[(w::C + NS) * 32] = 1.0;                 // the empty slot
  col[(w::G + NS) * 32] = 0.0;
  if (JAC) {
#pragma unroll
    for (int e = 0; e < NS * NS; ++e) Mx[((1 + e / NS) * N + 1 + e % NS) * 32] = 0.0;
  }
  const double Ctot = rho * S;
  const fx::i64 D = (fx::i64)((t.L + 128ull) >> 8) - m.lpr0;
  const fx::i64 shift = t.iT2 - t.L2;
  double* const Cc = col + w::C * 32;
  double* const Gc = col + w::G * 32;
  double* const wd = col + (uoff + 1) * 32;
  double* const Jm = Mx + (N + 1) * 32;              // row 1 (species 0), column 1

  // exponents and concentration products of an FxRate
  auto prepare = [&](const FxRate& R, const Slots& s, fx::i64& Xf, fx::i64& Xr) {
    Xf = exponent_f(R, t, shift);
    Xr = Xf + (__double_as_longlong(*at(Gc, s.p0)) + __double_as_longlong(*at(Gc, s.p1))) -
         (__double_as_longlong(*at(Gc, s.r0)) + __double_as_longlong(*at(Gc, s.r1)));
  };
  auto in_range = [&](fx::i64 Xf, fx::i64 Xr) { return t.fast && fx::exp2_in_range(Xf) && fx::exp2_in_range(Xr); };
  auto scatter = [&](const FxRate& R, double q) {
    const Slots s = slots(R.w);
    double *a0 = at(wd, s.r0), *a1 = at(wd, s.r1), *a2 = at(wd, s.p0), *a3 = at(wd, s.p1);
    const double v0 = fma(R.nu[0], q, *a0), v1 = fma(R.nu[1], q, *a1);
    const double v2 = fma(R.nu[2], q, *a2), v3 = fma(R.nu[3], q, *a3);
    *a0 = v0; *a1 = v1; *a2 = v2; *a3 = v3;
  };
  // Jacobian share of an FxRate with rate constants already times the collision partner: q and dq/dT
  // into the production rates, the slots' derivatives into d(wdot)/dC (negated)
  auto derivatives = [&](const FxRate& R, const Slots& s, double ka, double kb, double a0, double a1, double b0,
                         double b1, double q, double dqdT) {
    scatter(R, q);
    const Slots x = slots(R.w);
    const unsigned row[4] = {x.r0, x.r1, x.p0, x.p1};
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      double* y = at(col + w::DWDT * 32, row[i]);
      *y = fma(R.nu[i], dqdT, *y);
    }
    auto column = [&](unsigned sp, double d) {
      double v[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) v[i] = fma(-R.nu[i], d, *at(Jm, row[i] * N + sp));
#pragma unroll
      for (int i = 0; i < 4; ++i) *at(Jm, row[i] * N + sp) = v[i];
    };
    column(s.r0, ka * a1);
    if (s.r1 != NS * 256u) column(s.r1, ka * a0);
    column(s.p0, -kb * b1);
    if (s.p1 != NS * 256u) column(s.p1, -kb * b0);
  };
  auto dlnkf_of = [&](double b, double TaK) { return fma(TaK * t.invT, t.invT, b * t.invT); };
  auto dlnKc_of = [&](const Slots& s, int dnu) {
    const double* Hc = col + w::H * 32;
    double dH = *at(const_cast<double*>(Hc), s.p0) - *at(const_cast<double*>(Hc), s.r0);
    if (s.p1 != NS * 256u) dH += *at(const_cast<double*>(Hc), s.p1);
    if (s.r1 != NS * 256u) dH -= *at(const_cast<double*>(Hc), s.r1);
    if (dnu) dH -= (double)dnu;
    return dH * t.invT;
  };
  // d(wdot)/dC through the collision partners: X times the efficiencies of set tb
  auto partner_rows = [&](const FxRate& R, double X) {
    const double* ef = m.eff + R.tb * NS;
    const Slots x = slots(R.w);
    const unsigned row[4] = {x.r0, x.r1, x.p0, x.p1};
    for (int i = 0; i < 4; ++i) {
      if (R.nu[i] == 0.0) continue;
      const double nx = -R.nu[i] * X;
      double* y = at(Jm, row[i] * N);
#pragma unroll
      for (int mm = 0; mm < NS; ++mm) y[mm * 32] = fma(nx, ef[mm], y[mm * 32]);
    }
  };

  const FxRate* R = m.rate;
  // ---- plain reactions, two at a time: four independent exponentials hide the integer latency ----
  int j = 0;
  if (!JAC) {
    for (; j + 1 < m.n_plain; j += 2, R += 2) {
      const Slots s0 = slots(R[0].c), s1 = slots(R[1].c);
      fx::i64 Xf0, Xr0, Xf1, Xr1;
      prepare(R[0], s0, Xf0, Xr0);
      prepare(R[1], s1, Xf1, Xr1);
      if (R[0].dnu) Xr0 += (fx::i64)R[0].dnu * D;
      if (R[1].dnu) Xr1 += (fx::i64)R[1].dnu * D;
      double kf0 = fx::exp2_q52(Xf0, m.e2), kr0 = fx::exp2_q52(Xr0, m.e2);
      double kf1 = fx::exp2_q52(Xf1, m.e2), kr1 = fx::exp2_q52(Xr1, m.e2);
      const bool ok0 = in_range(Xf0, Xr0), ok1 = in_range(Xf1, Xr1);
      if (!(ok0 && ok1)) {
        double x = 0.0, y, z;
        if (!ok0) fx::slow_rate(m, Gc, 32, R[0].id, nullptr, T, fx::ln_inv_of(t), t.fast, 1.0, &kf0, &kr0, &x, &y, &z);
        if (!ok1) fx::slow_rate(m, Gc, 32, R[1].id, nullptr, T, fx::ln_inv_of(t), t.fast, 1.0, &kf1, &kr1, &x, &y, &z);
      }
      const double q0 = fma(kf0, *at(Cc, s0.r0) * *at(Cc, s0.r1), -(kr0 * (*at(Cc, s0.p0) * *at(Cc, s0.p1))));
      const double q1 = fma(kf1, *at(Cc, s1.r0) * *at(Cc, s1.r1), -(kr1 * (*at(Cc, s1.p0) * *at(Cc, s1.p1))));
      scatter(R[0], q0);
      scatter(R[1], q1);
    }
  }
  // ---- the rest of the plain ones, third-body and fall-off reactions (stored in that order) ----
  const int n2 = m.n_plain + m.n_tb, n3 = n2 + m.n_fo;
  for (; j < n3; ++j, ++R) {
    const Slots s = slots(R->c);
    fx::i64 Xf, Xr;
    prepare(*R, s, Xf, Xr);
    if (R->dnu) Xr += (fx::i64)R->dnu * D;
    const double a0 = *at(Cc, s.r0), a1 = *at(Cc, s.r1), b0 = *at(Cc, s.p0), b1 = *at(Cc, s.p1);
    double Mc = 1.0;
    if (j >= m.n_plain) Mc = partners<NS>(m, col, R->tb, Ctot);
    double dlnkf = JAC ? dlnkf_of(R->b, R->TaK) : 0.0;
    double kf = fx::exp2_q52(Xf, m.e2), kr = fx::exp2_q52(Xr, m.e2);
    double dMr = 0.0, dkfdM = 0.0, invKc = 0.0;   // (d kf/d[M]) / kf; d kf/d[M] and 1 / Kc of the FP64 form
    bool fastk = in_range(Xf, Xr);
    if (j >= n2 && fastk) {
      const FxTroe& F = m.troe[R->troe];
      const fx::i64 Xk = F.lnA0 + (fx::i64)(fx::umulhi3(F.b0, t.L) - fx::umulhi3(F.Ta0, t.iT)) + shift - Xf;
      double fac = 1.0, dl = 0.0;
      fastk = troe_fast<JAC>(m, F, t, Xk, Mc, dlnkf, &fac, &dl, &dMr);
      kf *= fac;
      kr *= fac;
      if (JAC && fastk) dlnkf = dl;
    }
    if (!fastk)
      fx::slow_rate(m, Gc, 32, R->id, j >= n2 ? m.troe + R->troe : nullptr, T, fx::ln_inv_of(t), t.fast, Mc, &kf,
                    &kr, &dlnkf, &dkfdM, &invKc);
    const bool third = j >= m.n_plain && j < n2;
    if (!JAC) {
      double q = fma(kf, a0 * a1, -(kr * (b0 * b1)));
      if (third) q *= Mc;
      scatter(*R, q);
    } else {
      const double rev = kr * (b0 * b1), net = fma(kf, a0 * a1, -rev);
      double dqdT = fma(net, dlnkf, rev * dlnKc_of(s, R->dnu));
      double q = net, ka = kf, kb = kr;
      if (third) { q *= Mc; dqdT *= Mc; ka *= Mc; kb *= Mc; }
      derivatives(*R, s, ka, kb, a0, a1, b0, b1, q, dqdT);
      if (third) partner_rows(*R, net);
      else if (j >= n2) partner_rows(*R, fastk ? dMr * net : dkfdM * fma(a0, a1, -(b0 * b1 * invKc)));
    }
  }
  // ---- reactions with three species on a side or more than four net species ----
  for (int i = 0; i < m.n_gen; ++i) general_reaction<NS, JAC>(m, col, Mx, m.reac[i], t, T, shift, D, Ctot, uoff);

  // species and temperature rows: f_k = W_k w_k / rho, f_0 = -T sum h/RT w / (rho cp/R)
  double Q = 0.0, r31 = 0.0, r32 = 0.0;
#pragma unroll
  for (int k = 0; k < NS; ++k) {
    const double wk = col[(uoff + 1 + k) * 32];
    const double h = col[(w::H + k) * 32];
    Q = fma(h, wk, Q);
    if (JAC) {
      r31 = fma(col[(w::CP + k) * 32], wk, r31);
      r32 = fma(h, col[(w::DWDT + k) * 32], r32);
      col[(w::WK + k) * 32] = wk;
    }
    col[(uoff + 1 + k) * 32] = m.W[k] * (wk * invrho);
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
#pragma unroll 2
  for (int k = 0; k < NS; ++k) {
    double s = 0.0;
#pragma unroll
    for (int mm = 0; mm < NS; ++mm) s = fma(Jm[(k * N + mm) * 32], col[(w::C + mm) * 32], s);
    Rh = fma(-col[(w::H + k) * 32], s, Rh);
    const double dk = -s - col[(w::WK + k) * 32];
    col[(w::RK + k) * 32] = dk * rS;
    Jm[(k * N - 1) * 32] = -(m.W[k] * invrho * fma(-dk, t.invT, col[(w::DWDT + k) * 32]));
  }
  const double TQ = T * Q, TRh = T * Rh;
  const double Qr = TQ * ircp;                 // -f_0
  Mx[0] = fma(fma(T, r32, r31) - Rh, ircp, Qr * fma(cps, t.invT, -dcps) * (rho * ircp));
  const double RhS = TRh * iS, cpS = __dmul_rn(cps, iS), Qrr = Qr * rho;
#pragma unroll 2
  for (int mm = 0; mm < NS; ++mm) {
    double s = 0.0;
#pragma unroll
    for (int k = 0; k < NS; ++k) s = fma(-col[(w::H + k) * 32], Jm[(k * N + mm) * 32], s);
    const double Hm = T * s;
    Jm[(mm - N) * 32] = m.invW[mm] * ircp * fma(-Qrr, col[(w::CP + mm) * 32] - cpS, fma(rho, Hm, -RhS));
  }
#pragma unroll 2
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
