// The integrator of small mechanisms for launches of few cells: L = 8 or 16 lanes per cell.
//
// What bounds it: the stiffest cell's chain of attempts.  One thread per cell (integrator_cell.cu)
// does the least work in all, but an attempt of one warp takes about 600 k cycles however many of
// its lanes are in use (an FP64 instruction occupies its sub-partition for 64 cycles), and a launch
// of fewer cells than 128 an SM leaves lanes without work for that long.  Here the lanes of a cell
// share its species, reactions, Jacobian entries and matrix rows; the rows stay in registers from the
// factorisation through the six solves, whose unknowns travel by shuffles.  A mixing layer of 4096
// H2 cells takes 21 ms instead of 48, a block of 10007 cells across a flame 4.2 instead of 10.2
// (cell_lanes).  What is left is the dependent FP64 chain of a cell: the sums over its species.
//
// A cell's result must not depend on the launch it is part of, so every operation and the order of
// every sum are those of the one-thread kernel: sums over species or reactions are formed by one
// lane, or by all lanes alike, in its order (the production rates and the Jacobian entries by gather
// programs in the order of its scatters, CoLayout).  The two kernels agree bit for bit.
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <algorithm>

#include "chem_internal.h"
#include "integrator_cell.cuh"

namespace chem {
namespace {

using cell::View;
using fx::rcp;

struct CoParams {
  FxLayout fx;
  CoLayout co;
  MechLayout lay;
  const unsigned char *fxblob, *coblob, *blob;
  int stride;                  // doubles of workspace per cell
  QueueParams q;
};

struct Program {
  const int *woff, *wterm, *eoff, *epos;
  const CoTerm* term;
  int n, nent;
};

// workspace of one cell (doubles)
template <int NS>
struct Co {
  static constexpr int N = NS + 1;
  static constexpr int Y = 0, U = N, YS = 7 * N, M = 8 * N, C = M + N * N, G = C + N, H = G + N, CP = H + NS,
                       WD = CP + NS, DW = WD + NS, RK = DW + NS, SV = RK + NS, Q = SV + NS;
  // then q [n], dq/dT [n] and the values of the gather programs
  static int total(const CoLayout& c) {
    const int t = Q + 2 * c.n + c.nval;
    return (t + 7) / 16 * 16 + 8;        // neighbouring cells half of the banks apart
  }
};

// Right-hand side f(T, y) into out[0 .. N), y the mass fractions, and with JAC the negated Jacobian
// into the matrix: cell::rhs spread over the L lanes of a cell.
template <int NS, int L, bool JAC>
__device__ __forceinline__ void co_rhs(const View& m, const Program& pg, double* ws, unsigned mask, int u, double T,
                                       const double* y, double p, double invp, double* out) {
  using w = Co<NS>;
  constexpr int N = w::N, RS = (NS + L - 1) / L;
  double *C = ws + w::C, *G = ws + w::G, *H = ws + w::H, *CP = ws + w::CP, *WD = ws + w::WD, *DW = ws + w::DW;
  double *RK = ws + w::RK, *SV = ws + w::SV, *q = ws + w::Q, *dq = q + pg.n, *val = dq + pg.n;
  const fx::Temp t = fx::temp_of(T, m, JAC);
  double c[RS];
#pragma unroll
  for (int r = 0; r < RS; ++r) {
    const int k = u + r * L;
    c[r] = 0.0;
    if (k >= NS) continue;
    c[r] = __dmul_rn(y[k], m.invW[k]);
    C[k] = c[r];
    if (t.fast) {
      const FxSpecies& s = m.sp[t.rg * NS + k];
      const fx::u64 B = 0x8000000000000000ull;
      fx::u64 g = (fx::u64)s.g[4], h = (fx::u64)s.h[4], cp = (fx::u64)s.c[4];   // biased
#pragma unroll
      for (int i = 3; i >= 0; --i) {
        const fx::u64 b = i ? B : 0ull;
        g = (fx::umulhi3(g, t.tau) + (fx::u64)(s.g[i] - t.tau2)) ^ b;
        h = (fx::umulhi3(h, t.tau) + (fx::u64)(s.h[i] - t.tau2)) ^ b;
        cp = (fx::umulhi3(cp, t.tau) + (fx::u64)(s.c[i] - t.tau2)) ^ b;
      }
      g += fx::umulhi3((fx::u64)s.ga6, t.iT) + fx::umulhi3((fx::u64)s.gl, t.L) - (fx::u64)(t.iT2 + t.L2);
      h += fx::umulhi3((fx::u64)s.ha6, t.iT) - (fx::u64)t.iT2;
      G[k] = __longlong_as_double((fx::i64)g);
      H[k] = fx::to_double((fx::i64)h, 52);
      CP[k] = fx::to_double((fx::i64)cp, 52);
      if (JAC) {
        fx::u64 dc = fx::biased((fx::i64)(((fx::u64)s.c[4] ^ B) << 2));
        dc = (fx::umulhi3(dc, t.tau) + (fx::u64)(s.c[3] * 3 - t.tau2)) ^ B;
        dc = (fx::umulhi3(dc, t.tau) + (fx::u64)(s.c[2] * 2 - t.tau2)) ^ B;
        dc = fx::umulhi3(dc, t.tau) + (fx::u64)(s.c[1] - t.tau2);
        SV[k] = fx::to_double((fx::i64)dc, 52 + (t.rg == 0 ? kFxR0 : kFxR1));
      }
    } else {
      const cell::Species64 s = cell::species64(m, NS, k, T);
      G[k] = s.g; H[k] = s.h; CP[k] = s.cp;
      if (JAC) SV[k] = s.dcp;
    }
  }
  __syncwarp(mask);
  double S = 0.0, cps = 0.0, dcps = 0.0;
#pragma unroll
  for (int k = 0; k < NS; ++k) {
    const double ck = C[k];
    S += ck;
    cps = fma(ck, CP[k], cps);
    if (JAC) dcps = fma(ck, SV[k], dcps);
  }
  const double RTS = RU * T * S;
  const double rho = p * rcp(RTS), invrho = RTS * invp;
  __syncwarp(mask);
#pragma unroll
  for (int r = 0; r < RS; ++r)
    if (u + r * L < NS) C[u + r * L] = rho * c[r];
  if (u == 0) {
    C[NS] = 1.0;                               // the empty slot
    G[NS] = 0.0;
  }
  __syncwarp(mask);
  const double Ctot = rho * S;
  const fx::i64 D = (fx::i64)((t.L + 128ull) >> 8) - m.lpr0;
  const fx::i64 shift = t.iT2 - t.L2;
  const int n2 = m.n_plain + m.n_tb;
  auto Gi = [&](unsigned s) { return __double_as_longlong(G[s]); };

  // the lanes' reactions, the fall-off ones (stored last) first
  for (int jj = u; jj < pg.n; jj += L) {
    const int j = pg.n - 1 - jj;
    const FxRate& R = m.rate[j];
    const unsigned r0 = R.c[0] >> 8, r1 = R.c[1] >> 8, p0 = R.c[2] >> 8, p1 = R.c[3] >> 8;
    const fx::i64 Xf = fx::exponent_f(R, t, shift);
    fx::i64 Xr = Xf + (Gi(p0) + Gi(p1)) - (Gi(r0) + Gi(r1));
    if (R.dnu) Xr += (fx::i64)R.dnu * D;
    const double a0 = C[r0], a1 = C[r1], b0 = C[p0], b1 = C[p1];
    const bool third = j >= m.n_plain && j < n2;
    double Mc = 1.0;
    if (j >= m.n_plain) {
      Mc = Ctot;
      const int e1 = m.effoff[R.tb + 1];
      for (int e = m.effoff[R.tb]; e < e1; ++e) Mc = fma(m.effv[e], C[m.effidx[e]], Mc);
    }
    double dlnkf = JAC ? fma(R.TaK * t.invT, t.invT, R.b * t.invT) : 0.0;
    double kf = fx::exp2_q52(Xf, m.e2), kr = fx::exp2_q52(Xr, m.e2);
    double dMr = 0.0, dkfdM = 0.0, invKc = 0.0;
    bool fastk = t.fast && fx::exp2_in_range(Xf) && fx::exp2_in_range(Xr);
    if (j >= n2 && fastk) {
      const FxTroe& F = m.troe[R.troe];
      const fx::i64 Xk = F.lnA0 + (fx::i64)(fx::umulhi3(F.b0, t.L) - fx::umulhi3(F.Ta0, t.iT)) + shift - Xf;
      double fac = 1.0, dl = 0.0;
      fastk = fx::troe_fast<JAC>(m, F, t, Xk, Mc, dlnkf, &fac, &dl, &dMr);
      kf *= fac;
      kr *= fac;
      if (JAC && fastk) dlnkf = dl;
    }
    if (!fastk) {
      double skf = kf, skr = kr, sdl = dlnkf;
      fx::slow_rate(m, G, 1, R.id, j >= n2 ? m.troe + R.troe : nullptr, T, t.fast, Mc, &skf, &skr, &sdl, &dkfdM, &invKc);
      kf = skf; kr = skr; dlnkf = sdl;
    }
    if (!JAC) {
      double v = fma(kf, a0 * a1, -(kr * (b0 * b1)));
      if (third) v *= Mc;
      q[j] = v;
    } else {
      const double rev = kr * (b0 * b1), net = fma(kf, a0 * a1, -rev);
      double dH = H[p0] - H[r0];
      if (p1 != NS) dH += H[p1];
      if (r1 != NS) dH -= H[r1];
      if (R.dnu) dH -= (double)R.dnu;
      double dqdT = fma(net, dlnkf, rev * (dH * t.invT));
      double v = net, ka = kf, kb = kr;
      if (third) { v *= Mc; dqdT *= Mc; ka *= Mc; kb *= Mc; }
      q[j] = v;
      dq[j] = dqdT;
      val[4 * j] = ka * a1;
      val[4 * j + 1] = ka * a0;
      val[4 * j + 2] = -kb * b1;
      val[4 * j + 3] = -kb * b0;
      if (j >= m.n_plain)
        val[4 * pg.n + j - m.n_plain] = third ? net : fastk ? dMr * net : dkfdM * fma(a0, a1, -(b0 * b1 * invKc));
    }
  }
  __syncwarp(mask);
  // production rates
#pragma unroll
  for (int r = 0; r < RS; ++r) {
    const int k = u + r * L;
    if (k >= NS) continue;
    double a = 0.0, b = 0.0;
    const int e1 = pg.woff[k + 1];
    for (int e = pg.woff[k]; e < e1; ++e) {
      const int tm = pg.wterm[e];
      const double nu = m.nu[tm & 15];
      a = fma(nu, q[tm >> 4], a);
      if (JAC) b = fma(nu, dq[tm >> 4], b);
    }
    WD[k] = a;
    if (JAC) DW[k] = b;
    out[1 + k] = m.W[k] * (a * invrho);
  }
  __syncwarp(mask);
  double Q = 0.0, r31 = 0.0, r32 = 0.0;
#pragma unroll
  for (int k = 0; k < NS; ++k) {
    const double wk = WD[k], h = H[k];
    Q = fma(h, wk, Q);
    if (JAC) {
      r31 = fma(CP[k], wk, r31);
      r32 = fma(h, DW[k], r32);
    }
  }
  const double ircp = rcp(rho * cps);         // 1 / (rho cp/R)
  if (u == 0) out[0] = -(T * Q) * ircp;
  if (!JAC) {
    __syncwarp(mask);
    return;
  }

  double* M = ws + w::M;
  double* Jm = M + N + 1;                      // row 1 (species 0), column 1
  for (int e = u; e < N * N; e += L) M[e] = 0.0;
  __syncwarp(mask);
  for (int e = u; e < pg.nent; e += L) {
    double a = 0.0;
    const int i1 = pg.eoff[e + 1];
    for (int i = pg.eoff[e]; i < i1; ++i) a = fma(val[pg.term[i].src], pg.term[i].coef, a);
    M[pg.epos[e]] = a;
  }
  __syncwarp(mask);
  // the chain rule of cell::rhs: rows, then columns
  const double iS = rcp(S);
  const double rS = invrho * iS;
  double col[RS];
#pragma unroll
  for (int r = 0; r < RS; ++r) {
    const int k = u + r * L;
    if (k >= NS) continue;
    double s = 0.0;
#pragma unroll
    for (int mm = 0; mm < NS; ++mm) s = fma(Jm[k * N + mm], C[mm], s);
    SV[k] = s;
    const double dk = -s - WD[k];
    RK[k] = dk * rS;
    Jm[k * N - 1] = -(m.W[k] * invrho * fma(-dk, t.invT, DW[k]));
    s = 0.0;
#pragma unroll
    for (int i = 0; i < NS; ++i) s = fma(-H[i], Jm[i * N + k], s);
    col[r] = s;
  }
  __syncwarp(mask);
  double Rh = 0.0;
#pragma unroll
  for (int k = 0; k < NS; ++k) Rh = fma(-H[k], SV[k], Rh);
  const double TQ = T * Q, TRh = T * Rh;
  const double Qr = TQ * ircp;                 // -f_0
  if (u == 0) M[0] = fma(fma(T, r32, r31) - Rh, ircp, Qr * fma(cps, t.invT, -dcps) * (rho * ircp));
  const double RhS = TRh * iS, cpS = __dmul_rn(cps, iS), Qrr = Qr * rho;
#pragma unroll
  for (int r = 0; r < RS; ++r) {
    const int mm = u + r * L;
    if (mm >= NS) continue;
    const double Hm = T * col[r];
    Jm[mm - N] = m.invW[mm] * ircp * fma(-Qrr, CP[mm] - cpS, fma(rho, Hm, -RhS));
  }
  for (int e = u; e < NS * NS; e += L) {
    const int k = e / NS, mm = e % NS;
    double* x = Jm + k * N + mm;
    *x = m.W[k] * m.invW[mm] * (RK[k] + *x);
  }
  __syncwarp(mask);
}

// One Rodas4 attempt (attempt of integrator_cell.cu): row r L + u of the matrix in lane u
template <int NS, int L>
__device__ __forceinline__ bool co_attempt(const View& m, const Program& pg, double* ws, unsigned mask, int u, double p,
                                           double invp, double h, double rtol, double atol, double* e2) {
  using w = Co<NS>;
  constexpr int N = w::N, R = (N + L - 1) / L;
  const double invh = rcp(h), ig = invh * (1.0 / kGamma);
  double *Y = ws + w::Y, *U = ws + w::U, *YS = ws + w::YS, *M = ws + w::M;
  co_rhs<NS, L, true>(m, pg, ws, mask, u, Y[0], Y + 1, p, invp, U);
  double a[R][N];
  int pos[R];                                  // logical row of a lane's row, -1 beyond the matrix
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const int i = u + r * L;
    pos[r] = i < N ? i : -1;
    const double* row = M + (i < N ? i : 0) * N;
#pragma unroll
    for (int j = 0; j < N; ++j) {
      a[r][j] = row[j];
      if (j == i) a[r][j] += ig;
    }
  }
  // the value of one of a lane's R rows, chosen by a run-time index
  auto pick = [&](const double (&x)[R], int r) {
    double v = x[0];
#pragma unroll
    for (int i = 1; i < R; ++i)
      if (r == i) v = x[i];
    return v;
  };
  int own[N];                                  // physical row of logical row k
  bool singular = false;
#pragma unroll
  for (int k = 0; k < N; ++k) {
    unsigned long long best = 0ull;
    int bi = 0x7fffffff;                       // logical row << 8 | physical row
#pragma unroll
    for (int r = 0; r < R; ++r) {
      if (pos[r] < k) continue;
      const unsigned long long key = pivot_key(a[r][k]);
      const int id = pos[r] << 8 | (u + r * L);
      if (key > best || (key == best && id < bi)) { best = key; bi = id; }
    }
#pragma unroll
    for (int o = L / 2; o > 0; o >>= 1) {
      const unsigned long long ob = __shfl_xor_sync(mask, best, o, L);
      const int oi = __shfl_xor_sync(mask, bi, o, L);
      if (ob > best || (ob == best && oi < bi)) { best = ob; bi = oi; }
    }
    if (best == 0ull) singular = true;
    const int pr = bi & 255, lp = bi >> 8, src = pr % L, rr = pr / L;
    own[k] = pr;
#pragma unroll
    for (int r = 0; r < R; ++r) {
      if (u + r * L == pr) pos[r] = k;
      else if (pos[r] == k) pos[r] = lp;
    }
    double x[R];
#pragma unroll
    for (int r = 0; r < R; ++r) x[r] = a[r][k];
    const double ip = rcp(__shfl_sync(mask, pick(x, rr), src, L));
    double l[R];
#pragma unroll
    for (int r = 0; r < R; ++r) {
      l[r] = a[r][k] * ip;
      if (u + r * L == pr) a[r][k] = ip;
      else if (pos[r] > k) a[r][k] = l[r];
    }
#pragma unroll
    for (int j = k + 1; j < N; ++j) {
#pragma unroll
      for (int r = 0; r < R; ++r) x[r] = a[r][j];
      const double uj = __shfl_sync(mask, pick(x, rr), src, L);
#pragma unroll
      for (int r = 0; r < R; ++r)
        if (pos[r] > k) a[r][j] = fma(-l[r], uj, a[r][j]);
    }
  }

#pragma unroll 1
  for (int s = 0; s < 6; ++s) {
    double* us = U + s * N;
    if (s > 0) {
      const double* ra = kRA[s];
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const int i = u + r * L;
        if (i >= N) continue;
        double v = Y[i];
        for (int j = 0; j < s; ++j) v = fma(ra[j], U[j * N + i], v);
        YS[i] = v;
      }
      __syncwarp(mask);
      co_rhs<NS, L, false>(m, pg, ws, mask, u, YS[0], YS + 1, p, invp, us);
    }
    double v[R], z[R];
#pragma unroll
    for (int r = 0; r < R; ++r) v[r] = u + r * L < N ? us[u + r * L] : 0.0;
    for (int j = 0; j < s; ++j) {
      const double c = kRC[s][j] * invh;
#pragma unroll
      for (int r = 0; r < R; ++r)
        if (u + r * L < N) v[r] = fma(c, U[j * N + u + r * L], v[r]);
    }
#pragma unroll
    for (int k = 0; k < N - 1; ++k) {
      const double x = __shfl_sync(mask, pick(v, own[k] / L), own[k] % L, L);
#pragma unroll
      for (int r = 0; r < R; ++r)
        if (pos[r] > k) v[r] = fma(-a[r][k], x, v[r]);
    }
#pragma unroll
    for (int k = N - 1; k >= 0; --k) {
#pragma unroll
      for (int r = 0; r < R; ++r) z[r] = a[r][k];
      const double x = __shfl_sync(mask, pick(v, own[k] / L) * pick(z, own[k] / L), own[k] % L, L);
#pragma unroll
      for (int r = 0; r < R; ++r)
        if (pos[r] < k) v[r] = fma(-a[r][k], x, v[r]);
      if (u == k % L) us[k] = x;
    }
    __syncwarp(mask);
  }
  double rr[R];
#pragma unroll
  for (int r = 0; r < R; ++r) {
    rr[r] = 0.0;
    const int i = u + r * L;
    if (i >= N) continue;
    const double y = Y[i];
    double v = y;
#pragma unroll
    for (int s = 0; s < 6; ++s) v = fma(kRM[s], U[s * N + i], v);
    const double sc = fma(rtol, fx::max_pos(fabs(y), fabs(v)), atol);
    rr[r] = U[5 * N + i] * rcp(sc);
    U[5 * N + i] = v;
  }
  double acc = 0.0;
#pragma unroll
  for (int i = 0; i < N; ++i) {
    const double x = __shfl_sync(mask, rr[i / L], i % L, L);
    acc = fma(x, x, acc);
  }
  *e2 = acc * (1.0 / N);
  return !singular;
}

__device__ __forceinline__ void stage(const unsigned char* src, unsigned char* dst, int bytes) {
  const int4* s = (const int4*)src;
  int4* d = (int4*)dst;
  for (int i = threadIdx.x; i < bytes / 16; i += blockDim.x) d[i] = __ldg(s + i);
}

template <int NS, int L>
__global__ void __launch_bounds__(256, 1) co_advance_kernel(const __grid_constant__ CoParams P) {
  using w = Co<NS>;
  constexpr int N = w::N, R = (N + L - 1) / L;
  extern __shared__ __align__(16) unsigned char smem[];
  if (P.q.ncells_dev && *P.q.ncells_dev == 0u) return;     // an empty fallback pass
  stage(P.fxblob, smem, P.fx.bytes);
  stage(P.coblob, smem + P.fx.bytes, P.co.bytes);
  __syncthreads();
  const View m = cell::bind(smem, P.fx, P.blob, &P.lay);
  const unsigned char* cs = smem + P.fx.bytes;
  const Program pg{(const int*)(cs + P.co.o_woff), (const int*)(cs + P.co.o_wterm), (const int*)(cs + P.co.o_eoff),
                   (const int*)(cs + P.co.o_epos), (const CoTerm*)(cs + P.co.o_term), P.co.n, P.co.nent};
  const int lane = threadIdx.x & 31, u = lane % L;
  const unsigned mask = (L == 32 ? 0xffffffffu : (1u << (L & 31)) - 1u) << (lane & ~(L - 1));
  double* ws = (double*)(smem + P.fx.bytes + P.co.bytes) + (size_t)(threadIdx.x / L) * P.stride;
  double* Y = ws + w::Y;
  auto dummy = [&] {
#pragma unroll
    for (int r = 0; r < R; ++r)
      if (u + r * L < N) Y[u + r * L] = u + r * L == 0 ? 1000.0 : 1.0 / NS;
  };
  dummy();
  __syncwarp();
  const long long total = P.q.ncells_dev ? min((long long)*P.q.ncells_dev, (long long)P.q.segs[0].ncells)
                                         : P.q.total_chunks;
  const unsigned long long t0 = P.q.budget_ns > 0 ? global_ns() : 0ull;
  const Segment* S = &P.q.segs[0];
  int64_t at = 0;
  bool active = false, exhausted = false;
  double dt = 1.0, rtol = 1e-6, atol = 1e-10, p = 1.0e6, invp = 1.0e-6, t = 0.0, h = 1.0, facmax = 6.0;
  int attempts = 0, nacc = 0, nrej = 0;

  for (;;) {
    // ---- cells without work claim the next ones of the queue (warp-wide) ----
    for (;;) {
      const unsigned need = __ballot_sync(0xffffffffu, u == 0 && !active && !exhausted);
      if (need == 0u) break;
      const int leader = __ffs(need) - 1;
      unsigned long long base = 0ull;
      if (lane == leader) {
        bool stop = false;                         // as in the one-thread kernel
        if (P.q.budget_ns > 0) {
          const unsigned long long el = global_ns() - t0;
          stop = el > P.q.budget_ns ||
                 (P.q.stop && el > P.q.min_ns && *(const volatile unsigned int*)P.q.stop != 0u);
        }
        base = stop ? ~0ull : atomicAdd(P.q.counter, (unsigned long long)__popc(need));
      }
      base = __shfl_sync(0xffffffffu, base, leader);
      if (!active && !exhausted) {
        const unsigned long long mine = base + (unsigned long long)__popc(need & ((1u << (lane - u)) - 1u));
        if (base == ~0ull || mine >= (unsigned long long)total) {
          exhausted = true;
        } else {
          S = segment_of(P.q, (long long)mine);
          at = cell_of(S, (long long)mine - S->chunk_begin, 0);
          p = S->p[at];
          double y[R];
          bool bad = !isfinite(p) || !(p > 0.0);
#pragma unroll
          for (int r = 0; r < R; ++r) {
            const int i = u + r * L;
            if (i >= N) continue;
            y[r] = i == 0 ? S->T[at] : S->Y[(int64_t)(i - 1) * S->ld + at];
            bad = bad || !isfinite(y[r]) || (i == 0 && !(y[r] > 0.0));
          }
          bad = __any_sync(mask, bad);
          if (bad) {                                  // the cell is left unchanged
            if (u == 0) {
              if (S->status) S->status[at] = (int8_t)CHEM_CELL_NONFINITE;
              if (S->nsub) S->nsub[at] = 0;
              if (S->nrej) S->nrej[at] = 0;
            }
            p = 1.0e6;
          } else {
#pragma unroll
            for (int r = 0; r < R; ++r)
              if (u + r * L < N) Y[u + r * L] = y[r];
            active = true;
            invp = 1.0 / p;
            dt = S->dt; rtol = S->rtol; atol = S->atol;
            t = 0.0; h = dt; facmax = 6.0;
            attempts = 0; nacc = 0; nrej = 0;
          }
        }
      }
      __syncwarp();
    }
    if (__all_sync(0xffffffffu, !active)) break;

    // ---- one attempt ----
    int status = CHEM_CELL_OK;
    bool stop = false, last = false, finished = false;
    if (active) {
      if (attempts >= P.q.max_steps) {
        stop = true; status = CHEM_CELL_MAX_STEPS;
      } else {
        if (h >= dt - t) { h = dt - t; last = true; }
        if (h < 1e-12 * dt) { stop = true; status = CHEM_CELL_H_UNDERFLOW; }
      }
    }
    const bool run = active && !stop;
    double e2 = 0.0;
    const bool ok = co_attempt<NS, L>(m, pg, ws, mask, u, p, invp, run ? h : dt, rtol, atol, &e2);
    if (run) {
      if (!ok) {
        stop = true; status = CHEM_CELL_SINGULAR_LU;
      } else {
        ++attempts;
        const double fac = fx::step_factor(e2, m.e2, m.rc, m.lg);
        if (e2 <= 1.0) {
#pragma unroll
          for (int r = 0; r < R; ++r)
            if (u + r * L < N) Y[u + r * L] = ws[w::U + 5 * N + u + r * L];
          ++nacc;
          if (last) {
            finished = true;
          } else {
            t += h;
            h = h * fmin(fac, facmax);
            facmax = 6.0;
          }
        } else {
          ++nrej;
          h = h * fac;
          facmax = 1.0;
        }
      }
    }
    if (active && (stop || finished)) {
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const int i = u + r * L;
        if (i == 0) S->T[at] = Y[0];
        else if (i < N) S->Y[(int64_t)(i - 1) * S->ld + at] = Y[i];
      }
      if (u == 0) {
        if (S->status) S->status[at] = (int8_t)status;
        if (S->nsub) S->nsub[at] = nacc;
        if (S->nrej) S->nrej[at] = nrej;
      }
      active = false;
      dummy();
    }
    __syncwarp();
  }
}

template <int NS, int L>
int advance_t(const chem_mech_s* m, const QueueParams& Q, int sms, int smem_max, int max_ctas, cudaStream_t stream) {
  CoParams P;
  P.fx = m->fx; P.co = m->co; P.lay = m->lay;
  P.fxblob = (const unsigned char*)m->d_fx; P.coblob = (const unsigned char*)m->d_co;
  P.blob = (const unsigned char*)m->d_blob;
  P.stride = Co<NS>::total(m->co);
  P.q = Q;
  const size_t fixed = (size_t)m->fx.bytes + m->co.bytes, per = (size_t)P.stride * 8 * (32 / L);
  int64_t warps = std::min<int64_t>(8, ((int64_t)smem_max - (int64_t)fixed) / (int64_t)per);
  // spread over the SMs
  const int ctas = max_ctas > 0 ? std::min(max_ctas, sms) : sms;
  const int64_t need = std::max<int64_t>(1, (Q.total_chunks + 32 / L - 1) / (32 / L));
  warps = std::min<int64_t>(warps, (need + ctas - 1) / ctas);
  const int64_t grid = std::min<int64_t>(ctas, (need + warps - 1) / warps);
  CHEM_CUDA_TRY(cudaFuncSetAttribute((co_advance_kernel<NS, L>), cudaFuncAttributeMaxDynamicSharedMemorySize, smem_max));
  co_advance_kernel<NS, L><<<(unsigned)grid, 32 * (unsigned)warps, fixed + per * (size_t)warps, stream>>>(P);
  CHEM_CUDA_TRY(cudaGetLastError());
  return CHEM_OK;
}

template <int NS>
int advance_l(const chem_mech_s* m, const QueueParams& Q, int lanes, int sms, int smem_max, int max_ctas,
              cudaStream_t stream) {
  return lanes == 16 ? advance_t<NS, 16>(m, Q, sms, smem_max, max_ctas, stream)
                     : advance_t<NS, 8>(m, Q, sms, smem_max, max_ctas, stream);
}

}  // namespace

// Lanes per cell for a launch of ncells cells on `ctas` SMs: 16, 8, or 1 for the one-thread kernel.
// Measured on 152 SMs (16 lanes / 8 lanes / one thread), H2 mixing layer with dt 1 us: 1000 cells
// 11.9 / 17.2 / 45 ms, 4096: 21.0 / 21.2 / 47.8, 10007: 39.6 / 36.3 / 49, 20011: 70 / 60.3 / 54.6;
// flame fronts, dt 0.5 us: 333: 2.3 / 3.1 / 8.5, 4864: 3.0 / 3.8 / 10.2, 10007: 4.6 / 4.2 / 10.2,
// 20011: 7.7 / 6.7 / 10.3.  The lines are where the mixing layer's curves cross; the fronts, whose
// stiff cells are fewer, would gain beyond them.
int cell_lanes(const chem_mech_s* m, int64_t ncells, int ctas, int smem_max) {
  if (!m->co.bytes) return 1;
  const int lanes = ncells <= 28 * (int64_t)ctas ? 16 : ncells <= 104 * (int64_t)ctas ? 8 : 1;
  int stride = 0;
  switch (m->ns) {
    case 8: stride = Co<8>::total(m->co); break;
    case 9: stride = Co<9>::total(m->co); break;
    case 10: stride = Co<10>::total(m->co); break;
    case 11: stride = Co<11>::total(m->co); break;
    default: return 1;
  }
  // room for at least half of the warps, else the one-thread kernel, which needs less per reaction
  return m->fx.bytes + m->co.bytes + 4ll * (32 / lanes) * stride * 8 <= smem_max ? lanes : 1;
}

int launch_coop_advance(const chem_mech_s* m, const QueueParams& Q, int lanes, int sms, int smem_max, int max_ctas,
                        cudaStream_t stream) {
  switch (m->ns) {
    case 8: return advance_l<8>(m, Q, lanes, sms, smem_max, max_ctas, stream);
    case 9: return advance_l<9>(m, Q, lanes, sms, smem_max, max_ctas, stream);
    case 10: return advance_l<10>(m, Q, lanes, sms, smem_max, max_ctas, stream);
    case 11: return advance_l<11>(m, Q, lanes, sms, smem_max, max_ctas, stream);
    default: set_error("no cell kernel for %d species", m->ns); return CHEM_EINVAL;
  }
}

}  // namespace chem
