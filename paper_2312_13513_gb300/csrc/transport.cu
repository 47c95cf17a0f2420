// Thermophysical and transport properties per cell on sm_103a (the paper's Thermo class, §3.1:
// "Newton's method and high-order temperature polynomials", compute bound).
//
// * chem_mixture_thermo: mixture h and cp from the NASA-7 polynomials (one thread per cell).
// * chem_temperature_from_enthalpy: T from h by Newton on the same polynomials (one thread per
//   cell; |dT| < 1e-9 T within 50 iterations and T in [200, 6000] K, else status 1 and T
//   unchanged).
// * chem_transport_eval: mixture-averaged viscosity (Wilke), conductivity (Mathur-Saxena) and
//   diffusion coefficients D_km = (1 - Y_k) / sum_{j != k} X_j / D_jk from cubic fits in ln T.
//   The FP64 pipe bounds it (19 SM cycles a warp instruction), so
//   - the fits and their exponentials run in fixed point on the integer pipe (fixed.cuh): no FP64
//     instruction per pair instead of 13;
//   - Wilke's sum is expanded: with s = mu^(1/2), sum_j X_j (1 + s_k wq_jk / s_j)^2 cw_kj =
//     sum_j cw_kj X_j + 2 s_k sum_j (cw wq)_kj X_j / s_j + s_k^2 sum_j (cw wq^2)_kj X_j / s_j^2, three
//     matrix-vector products with constant matrices: 3 FP64 instructions a pair instead of 5 (all
//     terms have one sign for non-negative X, nothing cancels);
//   - small mechanisms (ns <= 15) take one thread per cell, with the cell's vectors in a warp's
//     interleaved shared memory (conflict-free, no shuffles, no idle lanes); a binary coefficient
//     joins both species' sums when it is made, so that 45 values a cell are stored instead of 72
//     and up to sixteen warps share an SM (100003 H2 cells 170 -> 131 us, 2^20 1395 -> 1122 us);
//     larger mechanisms take a warp per cell, lanes over species and pairs.
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <algorithm>
#include <cmath>
#include <limits>
#include <vector>

#include "chem_internal.h"
#include "fixed.cuh"
#include "fx_rates.cuh"
#include "thermo.cuh"

using namespace chem;

struct chem_transport_s {
  chem_mech_s* mech = nullptr;
  int ns = 0;
  double* d = nullptr;                 // one device allocation holding the tables below
  const double* mu_poly = nullptr;     // [ns][4]
  const double* lam_poly = nullptr;    // [ns][4]
  const double* diff_poly = nullptr;   // [ns][ns][4]
  const double* invW = nullptr;        // [ns]
  // Wilke's constants cw wq^i, i = 0, 1, 2, of the pair (k, j) at [(i * ns + j) * ns + k], with
  // wq = (W_j / W_k)^(1/4) and cw = (8 (1 + W_k / W_j))^(-1/2)
  const double* wilke = nullptr;
  const int* pairs = nullptr;          // [ns (ns - 1) / 2]: j | k << 16, j < k, row-major upper triangle
  // the fits as base-2 exponents, cubic in log2(T) / 16, Q11.52 with the leading coefficient biased
  // (fixed.cuh): mu / 2 and lambda per species, -D per pair; null where a coefficient does not fit
  const long long *mu_fx = nullptr, *lam_fx = nullptr, *diff_fx = nullptr;
};

namespace {

constexpr double kPatm = 1.01325e6;

// The FP64 pipe bounds these kernels (about 13 FP64 instructions a species); with the species
// polynomials in fixed point two are left: h and cp of 100003 cells, H2 29 -> 13 us, CH4 142 -> 55 us,
// T from h (guess 2 % off) 115 -> 39 and 424 -> 130 us.  Errors against extended precision are no
// larger than the FP64 form's (5e-16 and 1.2e-15 of sum |h|, against 3.4e-15 and 1.4e-15).
__global__ void __launch_bounds__(128) mixture_thermo_kernel(const unsigned char* blob, MechLayout L,
                                                             const FxEnthalpy* hk, const double* T, const double* Y,
                                                             int64_t ld, int64_t n, double* h, double* cp) {
  for (int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; c < n; c += (int64_t)gridDim.x * blockDim.x) {
    double hh, cc;
    const Tau q = tau_of(T[c]);
    if (hk && q.fast) {
      hh = 0.0;
      cc = 0.0;
      const FxEnthalpy* E = hk + q.rg * L.ns;
#pragma unroll 3
      for (int k = 0; k < L.ns; ++k) {
        const double y = Y[(int64_t)k * ld + c];
        hh = fma(y, fx_enthalpy(E[k], q), hh);
        cc = fma(y, fx_cp(E[k], q), cc);
      }
      hh *= RU;
      cc *= RU;
    } else {
      h_cp_mass(blob, L, T[c], Y, ld, c, nullptr, &hh, &cc);
    }
    if (h) h[c] = hh;
    if (cp) cp[c] = cc;
  }
}

__global__ void __launch_bounds__(128) temperature_from_h_kernel(const unsigned char* blob, MechLayout L,
                                                                 const FxEnthalpy* hk, const double* h0,
                                                                 const double* Y, int64_t ld, int64_t n, double* T,
                                                                 int8_t* status) {
  for (int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; c < n; c += (int64_t)gridDim.x * blockDim.x) {
    const double target = h0[c];
    double Tn = T[c];
    bool conv = false;
    if (isfinite(target) && Tn >= 200.0 && Tn <= 6000.0) {
      const double tr = target * (1.0 / RU);
      for (int it = 0; it < 50; ++it) {
        double dT;
        const Tau q = tau_of(Tn);
        // cp only scales the step: FP32, where its magnitude allows
        double hs = 0.0;
        float cs = 0.0f;
        if (hk && q.fast) {
          const FxEnthalpy* E = hk + q.rg * L.ns;
#pragma unroll 3
          for (int k = 0; k < L.ns; ++k) {
            const double y = Y[(int64_t)k * ld + c];
            hs = fma(y, fx_enthalpy(E[k], q), hs);
            cs = fmaf(f32_of(y), cp_f32(E[k], q), cs);
          }
        }
        if (cs > 1e-30f && cs < 1e30f) {
          dT = (hs - tr) * f64_of(1.0f / cs);
        } else {
          double hh, cp;
          h_cp_mass(blob, L, Tn, Y, ld, c, nullptr, &hh, &cp);
          dT = (hh - target) / cp;
        }
        Tn -= dT;
        if (!in_bounds(Tn, 200.0, 6000.0)) break;
        if (less_abs(dT, 1e-9 * Tn)) { conv = true; break; }
      }
    }
    if (conv) T[c] = Tn;
    if (status) status[c] = conv ? 0 : 1;
  }
}

struct TrParams {
  const double *T, *p, *Y;
  int64_t ld, n;
  double *mu, *lam, *Dm;
  const double *mu_poly, *lam_poly, *diff_poly, *invW, *wilke;
  const int* pairs;
  const long long *mu_fx, *lam_fx, *diff_fx;
  const fx::u64 *e2, *lg;
  const uint32_t* rc;
  int ns;
};

// index of the unordered pair (j, k), j < k, in the row-major upper triangle
__device__ __forceinline__ int pair_index(int j, int k, int ns) { return j * ns - (j * (j + 1)) / 2 + (k - j - 1); }

__device__ __forceinline__ double poly3(const double* c, double x) {
  return __ldg(c) + x * (__ldg(c + 1) + x * (__ldg(c + 2) + x * __ldg(c + 3)));
}

// Temperature of a cell: in fixed point log2(T) / 16 (Q0.64) for T in [1, 65536), otherwise ln T
struct FitT {
  bool fast;
  fx::u64 l;
  fx::i64 l2;
  double lnT;
};

__device__ __forceinline__ FitT fit_t(double T, const TrParams& P) {
  FitT t;
  t.fast = P.mu_fx && (unsigned)__double2hiint(T) - 0x3ff00000u < 0x40f00000u - 0x3ff00000u;
  int e;
  const fx::u64 m = fx::mantissa(t.fast ? T : 1024.0, e);
  const fx::u64 L = ((fx::u64)e << 60) + fx::log2_mant_q60(m, P.rc, P.lg);
  t.l = e == 0 && (fx::i64)L < 0 ? 0ull : L;               // a few units below zero at T = 1
  t.l2 = (fx::i64)(t.l >> 1);
  t.lnT = t.fast ? 0.0 : log(T);
  return t;
}

// a fit's base-2 exponent at t: c = 4 coefficients in fixed point
__device__ __forceinline__ fx::i64 fit_x(const long long* c, const FitT& t) {
  const fx::u64 B = 0x8000000000000000ull;
  fx::u64 a = (fx::umulhi3((fx::u64)c[3], t.l) + (fx::u64)(c[2] - t.l2)) ^ B;
  a = (fx::umulhi3(a, t.l) + (fx::u64)(c[1] - t.l2)) ^ B;
  return (fx::i64)(fx::umulhi3(a, t.l) + (fx::u64)(c[0] - t.l2));
}
__device__ __forceinline__ double exp2_any(fx::i64 X, const fx::u64* e2) {
  return fx::exp2_in_range(X) ? fx::exp2_q52(X, e2) : exp(fx::to_double(X, 52) * fx::kLn2);
}

// mu^(1/2) and its inverse, lambda and its inverse, of species k
__device__ __forceinline__ void pure_species(const TrParams& P, const long long* mu_fx, const long long* lam_fx,
                                             const fx::u64* e2, const FitT& t, int k, double& s, double& is, double& l,
                                             double& il) {
  if (t.fast) {
    const fx::i64 x = fit_x(mu_fx + 4 * k, t), y = fit_x(lam_fx + 4 * k, t);
    s = exp2_any(x, e2); is = exp2_any(-x, e2);
    l = exp2_any(y, e2); il = exp2_any(-y, e2);
  } else {
    const double x = 0.5 * poly3(P.mu_poly + 4 * k, t.lnT), y = poly3(P.lam_poly + 4 * k, t.lnT);
    s = exp(x); is = exp(-x);
    l = exp(y); il = exp(-y);
  }
}

// D_km from its sum; 1 / D_jk(p) = pr / D_jk(p_atm).  A cell holding species k alone takes the
// self-diffusion fit.
__device__ __forceinline__ double mixture_d(const TrParams& P, double dsum, double y, double pr, double T, int k) {
  if (dsum > 0.0) return (1.0 - y) * fx::rcp(dsum * pr);
  return exp(poly3(P.diff_poly + 4 * (k * P.ns + k), log(T))) / pr;
}

// One thread per cell (ns <= 15).  Shared memory: exp2 table, the fits and Wilke's constants (read
// by warp-uniform addresses), then per warp the cells' vectors, element e of a lane at e * 32.
__global__ void __launch_bounds__(512, 1) transport_cell_kernel(const TrParams P) {
  extern __shared__ __align__(16) double tsm[];
  const int ns = P.ns, npair = ns * (ns - 1) / 2;
  fx::u64* e2 = (fx::u64*)tsm;
  long long* mu_fx = (long long*)(tsm + 256);
  long long* lam_fx = mu_fx + 4 * ns;
  long long* diff_fx = lam_fx + 4 * ns;
  double* wk = (double*)(diff_fx + 4 * npair);
  double* invW = wk + 3 * ns * ns;
  for (int i = threadIdx.x; i < 256; i += blockDim.x) e2[i] = P.e2[i];
  for (int i = threadIdx.x; i < 4 * ns && P.mu_fx; i += blockDim.x) { mu_fx[i] = P.mu_fx[i]; lam_fx[i] = P.lam_fx[i]; }
  for (int i = threadIdx.x; i < 4 * npair && P.mu_fx; i += blockDim.x) diff_fx[i] = P.diff_fx[i];
  for (int i = threadIdx.x; i < 3 * ns * ns; i += blockDim.x) wk[i] = P.wilke[i];
  for (int i = threadIdx.x; i < ns; i += blockDim.x) invW[i] = P.invW[i];
  __syncthreads();
  const int lane = threadIdx.x & 31;
  double* X = invW + ns + (ns & 1) + (size_t)(threadIdx.x >> 5) * 5 * ns * 32 + lane;   // mole fractions
  double* X1 = X + ns * 32;                  // X / s
  double* X2 = X1 + ns * 32;                 // X / s^2
  double* s = X2 + ns * 32;                  // mu_k^(1/2)
  double* Ds = s + ns * 32;                  // sum_j X_j / D_jk(p_atm)
  for (int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; c < P.n; c += (int64_t)gridDim.x * blockDim.x) {
    const double T = P.T[c];
    const FitT t = fit_t(T, P);
    const double pr = P.p[c] / kPatm;
    double S = 0.0;
    for (int k = 0; k < ns; ++k) {
      const double x = P.Y[(int64_t)k * P.ld + c] * invW[k];
      X[k * 32] = x;
      S += x;
    }
    const double iS = 1.0 / S;
    double lx = 0.0, lxi = 0.0;
#pragma unroll 2
    for (int k = 0; k < ns; ++k) {
      double sk, is, l, il;
      pure_species(P, mu_fx, lam_fx, e2, t, k, sk, is, l, il);
      const double x = X[k * 32] * iS;
      const double x1 = x * is;
      X[k * 32] = x;
      X1[k * 32] = x1;
      X2[k * 32] = x1 * is;
      s[k * 32] = sk;
      lx = fma(x, l, lx);
      lxi = fma(x, il, lxi);
    }
    if (P.Dm) {
      // the unordered pairs row by row: a coefficient joins both species' sums at once, so that a sum
      // per species is stored instead of a coefficient per pair
      for (int k = 0; k < ns; ++k) Ds[k * 32] = 0.0;
      int q = 0;
      for (int j = 0; j < ns; ++j) {
        const double xj = X[j * 32];
        double sum = Ds[j * 32];
        if (t.fast) {
#pragma unroll 4
          for (int k = j + 1; k < ns; ++k, ++q) {
            const double e = exp2_any(fit_x(diff_fx + 4 * q, t), e2);       // 1 / D_jk(p_atm)
            sum = fma(X[k * 32], e, sum);
            Ds[k * 32] = fma(xj, e, Ds[k * 32]);
          }
        } else {
          for (int k = j + 1; k < ns; ++k) {
            const double e = exp(-poly3(P.diff_poly + 4 * (j * ns + k), t.lnT));
            sum = fma(X[k * 32], e, sum);
            Ds[k * 32] = fma(xj, e, Ds[k * 32]);
          }
        }
        P.Dm[(int64_t)j * P.ld + c] = mixture_d(P, sum, P.Y[(int64_t)j * P.ld + c], pr, T, j);
      }
    }
    double num = 0.0;
    for (int k = 0; k < ns; ++k) {
      double a = 0.0, b = 0.0, d = 0.0;
      if (P.mu) {
#pragma unroll 3
        for (int j = 0; j < ns; ++j) {
          a = fma(wk[j * ns + k], X[j * 32], a);
          b = fma(wk[(ns + j) * ns + k], X1[j * 32], b);
          d = fma(wk[(2 * ns + j) * ns + k], X2[j * 32], d);
        }
        const double sk = s[k * 32];
        const double den = fma(sk, fma(sk, d, b + b), a);
        num = fma(X[k * 32] * sk, sk * fx::rcp(den), num);
      }
    }
    if (P.mu) P.mu[c] = num;
    if (P.lam) P.lam[c] = 0.5 * (lx + fx::rcp(lxi));
  }
}

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// One warp per cell: lanes over species, and over pairs for the binary coefficients
__global__ void __launch_bounds__(256) transport_warp_kernel(const TrParams P) {
  extern __shared__ __align__(16) double tsm[];
  const int ns = P.ns, npair = ns * (ns - 1) / 2;
  fx::u64* e2 = (fx::u64*)tsm;
  for (int i = threadIdx.x; i < 256; i += blockDim.x) e2[i] = P.e2[i];
  __syncthreads();
  const int lane = threadIdx.x & 31, wpb = blockDim.x >> 5;
  double* X = tsm + 256 + (size_t)(threadIdx.x >> 5) * (4 * ns + npair);   // as transport_cell_kernel
  double* X1 = X + ns;
  double* X2 = X1 + ns;
  double* s = X2 + ns;
  double* E = s + ns;
  for (int64_t c = (int64_t)blockIdx.x * wpb + (threadIdx.x >> 5); c < P.n; c += (int64_t)gridDim.x * wpb) {
    const double T = P.T[c];
    const FitT t = fit_t(T, P);
    const double pr = P.p[c] / kPatm;
    double yw = 0.0;
    for (int k = lane; k < ns; k += 32) {
      const double x = P.Y[(int64_t)k * P.ld + c] * __ldg(P.invW + k);
      X[k] = x;
      yw += x;
    }
    const double iS = fx::rcp(warp_sum(yw));
    double lx = 0.0, lxi = 0.0;
    for (int k = lane; k < ns; k += 32) {
      double sk, is, l, il;
      pure_species(P, P.mu_fx, P.lam_fx, e2, t, k, sk, is, l, il);
      const double x = X[k] * iS;
      const double x1 = x * is;
      X[k] = x;
      X1[k] = x1;
      X2[k] = x1 * is;
      s[k] = sk;
      lx = fma(x, l, lx);
      lxi = fma(x, il, lxi);
    }
    if (P.lam) {
      lx = warp_sum(lx);
      lxi = warp_sum(lxi);
      if (lane == 0) P.lam[c] = 0.5 * (lx + fx::rcp(lxi));
    }
    if (P.Dm) {
      if (t.fast) {
#pragma unroll 2
        for (int q = lane; q < npair; q += 32) {
          const longlong2 c01 = __ldg(reinterpret_cast<const longlong2*>(P.diff_fx + 4 * q));
          const longlong2 c23 = __ldg(reinterpret_cast<const longlong2*>(P.diff_fx + 4 * q + 2));
          const long long cc[4] = {c01.x, c01.y, c23.x, c23.y};
          E[q] = exp2_any(fit_x(cc, t), e2);
        }
      } else {
        for (int q = lane; q < npair; q += 32) {
          const int jk = __ldg(P.pairs + q);
          E[q] = exp(-poly3(P.diff_poly + 4 * ((jk & 0xffff) * ns + (jk >> 16)), t.lnT));
        }
      }
    }
    __syncwarp();
    double num = 0.0;
    for (int k = lane; k < ns; k += 32) {
      double a = 0.0, b = 0.0, d = 0.0, dsum = 0.0;
      const double* w0 = P.wilke + k;
      const double* w1 = w0 + ns * ns;
      const double* w2 = w1 + ns * ns;
      int q = k - 1;                         // pair_index(j, k) for j < k, then of (k, j)
#pragma unroll 4
      for (int j = 0; j < ns; ++j) {
        const double x = X[j];
        a = fma(__ldg(w0 + j * ns), x, a);
        b = fma(__ldg(w1 + j * ns), X1[j], b);
        d = fma(__ldg(w2 + j * ns), X2[j], d);
        if (P.Dm) {
          dsum = fma(x, j == k ? 0.0 : E[q], dsum);
          q += j < k - 1 ? ns - 2 - j : (j == k - 1 ? 0 : (j == k ? 0 : 1));
          if (j == k) q = pair_index(k, k + 1, ns);
        }
      }
      const double sk = s[k];
      const double den = fma(sk, fma(sk, d, b + b), a);
      num = fma(X[k] * sk, sk * fx::rcp(den), num);
      if (P.Dm) P.Dm[(int64_t)k * P.ld + c] = mixture_d(P, dsum, P.Y[(int64_t)k * P.ld + c], pr, T, k);
    }
    if (P.mu) {
      num = warp_sum(num);
      if (lane == 0) P.mu[c] = num;
    }
    __syncwarp();
  }
}

inline unsigned grid_cells(int64_t n, int per_block) {
  return (unsigned)std::max<int64_t>(1, std::min<int64_t>((n + per_block - 1) / per_block, 152 * 16));
}

}  // namespace

extern "C" int chem_mixture_thermo(chem_mech_t m, const double* T, const double* Y, int64_t ld, int64_t ncells,
                                   double* h, double* cp, chem_stream_t stream) {
  if (!m || ncells < 0 || ld < ncells) { set_error("bad arguments"); return CHEM_EINVAL; }
  if (ncells == 0) return CHEM_OK;
  if (!T || !Y || (!h && !cp)) { set_error("NULL pointer"); return CHEM_EINVAL; }
  mixture_thermo_kernel<<<grid_cells(ncells, 128), 128, 0, (cudaStream_t)stream>>>(
      (const unsigned char*)m->d_blob, m->lay, m->d_hk, T, Y, ld, ncells, h, cp);
  CHEM_CUDA_TRY(cudaGetLastError());
  return CHEM_OK;
}

extern "C" int chem_temperature_from_enthalpy(chem_mech_t m, const double* h, const double* Y, int64_t ld,
                                              int64_t ncells, double* T, int8_t* status, chem_stream_t stream) {
  if (!m || ncells < 0 || ld < ncells) { set_error("bad arguments"); return CHEM_EINVAL; }
  if (ncells == 0) return CHEM_OK;
  if (!h || !Y || !T) { set_error("NULL pointer"); return CHEM_EINVAL; }
  temperature_from_h_kernel<<<grid_cells(ncells, 128), 128, 0, (cudaStream_t)stream>>>(
      (const unsigned char*)m->d_blob, m->lay, m->d_hk, h, Y, ld, ncells, T, status);
  CHEM_CUDA_TRY(cudaGetLastError());
  return CHEM_OK;
}

extern "C" int chem_transport_free(chem_transport_t t) {
  if (!t) { set_error("NULL transport"); return CHEM_EINVAL; }
  if (t->d) cudaFree(t->d);
  delete t;
  return CHEM_OK;
}

extern "C" int chem_transport_create(chem_mech_t m, const chem_transport_desc* d, chem_transport_t* out) {
  if (!m || !d || !out) { set_error("NULL argument"); return CHEM_EINVAL; }
  *out = nullptr;
  const int ns = d->n_species;
  if (ns != m->ns || !d->mu_poly || !d->lambda_poly || !d->diff_poly) {
    set_error("transport data do not match the mechanism (ns %d vs %d) or a table is NULL", ns, m->ns);
    return CHEM_EINVAL;
  }
  const size_t n1 = (size_t)ns * 4, n2 = (size_t)ns * ns * 4, nw = (size_t)ns * ns;
  const size_t npair = (size_t)ns * (ns - 1) / 2;
  for (size_t i = 0; i < n1; ++i) {
    if (!std::isfinite(d->mu_poly[i]) || !std::isfinite(d->lambda_poly[i])) {
      set_error("non-finite transport fit");
      return CHEM_EINVAL;
    }
  }
  // one buffer of 8-byte words: the FP64 tables, the pair list (as ints), the fixed-point fits
  const size_t o_lam = n1, o_diff = 2 * n1, o_invw = o_diff + n2, o_wilke = o_invw + ns, o_pairs = o_wilke + 3 * nw;
  const size_t o_fx = (o_pairs + (npair + 1) / 2 + 1) & ~(size_t)1;      // 16-byte aligned
  std::vector<double> h(o_fx + 2 * n1 + 4 * npair);
  double* p = h.data();
  std::copy(d->mu_poly, d->mu_poly + n1, p);
  std::copy(d->lambda_poly, d->lambda_poly + n1, p + o_lam);
  std::copy(d->diff_poly, d->diff_poly + n2, p + o_diff);
  for (int k = 0; k < ns; ++k) p[o_invw + k] = 1.0 / m->W[k];
  for (int j = 0; j < ns; ++j)
    for (int k = 0; k < ns; ++k) {
      const double wq = std::pow(m->W[j] / m->W[k], 0.25), cw = 1.0 / std::sqrt(8.0 * (1.0 + m->W[k] / m->W[j]));
      p[o_wilke + (size_t)j * ns + k] = cw;
      p[o_wilke + nw + (size_t)j * ns + k] = cw * wq;
      p[o_wilke + 2 * nw + (size_t)j * ns + k] = cw * wq * wq;
    }
  int* pairs = reinterpret_cast<int*>(p + o_pairs);
  for (int j = 0, q = 0; j < ns; ++j)
    for (int k = j + 1; k < ns; ++k) pairs[q++] = j | (k << 16);
  // f * poly(ln T) / ln 2 in powers of log2(T) / 16; no partial sum can leave Q11.52 where the
  // coefficients' magnitudes sum to at most 2000
  bool fits = true;
  long long* fxw = reinterpret_cast<long long*>(p + o_fx);
  const long double l2 = std::log(2.0L);
  auto fixed = [&](const double* c, double f, long long* o) {
    long double scale = 1.0L / l2, sum = 0.0L;
    for (int i = 0; i < 4; ++i, scale *= 16.0L * l2) {
      const long double v = (long double)f * c[i] * scale;
      sum += std::fabs(v);
      o[i] = std::fabs(v) <= 2000.0L ? (long long)std::nearbyintl(v * 4503599627370496.0L) : 0;
    }
    o[3] = (long long)fx::biased(o[3]);
    if (!(sum <= 2000.0L)) fits = false;
  };
  for (int k = 0; k < ns; ++k) {
    fixed(d->mu_poly + 4 * k, 0.5, fxw + 4 * k);
    fixed(d->lambda_poly + 4 * k, 1.0, fxw + n1 + 4 * k);
  }
  for (size_t q = 0; q < npair; ++q)
    fixed(d->diff_poly + 4 * ((size_t)(pairs[q] & 0xffff) * ns + (pairs[q] >> 16)), -1.0, fxw + 2 * n1 + 4 * q);
  chem_transport_s* t = new chem_transport_s();
  t->mech = m;
  t->ns = ns;
  cudaError_t e = cudaMalloc((void**)&t->d, h.size() * sizeof(double));
  if (e == cudaSuccess) e = cudaMemcpy(t->d, h.data(), h.size() * sizeof(double), cudaMemcpyHostToDevice);
  if (e != cudaSuccess) {
    const int rc = cuda_fail(e, "transport tables");
    chem_transport_free(t);
    return rc;
  }
  t->mu_poly = t->d;
  t->lam_poly = t->d + o_lam;
  t->diff_poly = t->d + o_diff;
  t->invW = t->d + o_invw;
  t->wilke = t->d + o_wilke;
  t->pairs = reinterpret_cast<const int*>(t->d + o_pairs);
  if (fits) {
    t->mu_fx = reinterpret_cast<const long long*>(t->d + o_fx);
    t->lam_fx = t->mu_fx + n1;
    t->diff_fx = t->mu_fx + 2 * n1;
  }
  *out = t;
  return CHEM_OK;
}

extern "C" int chem_transport_eval(chem_transport_t t, const double* T, const double* p, const double* Y,
                                   int64_t ld, int64_t ncells, double* mu, double* lambda, double* Dmix,
                                   chem_stream_t stream) {
  if (!t || ncells < 0 || ld < ncells) { set_error("bad arguments"); return CHEM_EINVAL; }
  if (ncells == 0) return CHEM_OK;
  if (!T || !p || !Y || (!mu && !lambda && !Dmix)) { set_error("NULL pointer"); return CHEM_EINVAL; }
  TrParams P;
  P.T = T; P.p = p; P.Y = Y; P.ld = ld; P.n = ncells; P.mu = mu; P.lam = lambda; P.Dm = Dmix;
  P.mu_poly = t->mu_poly; P.lam_poly = t->lam_poly; P.diff_poly = t->diff_poly; P.invW = t->invW;
  P.wilke = t->wilke; P.pairs = t->pairs; P.ns = t->ns;
  P.mu_fx = t->mu_fx; P.lam_fx = t->lam_fx; P.diff_fx = t->diff_fx;
  P.e2 = t->mech->d_e2; P.lg = t->mech->d_lg; P.rc = t->mech->d_rc;
  const int ns = t->ns, npair = ns * (ns - 1) / 2;
  int dev = 0, sms = 0;
  CHEM_CUDA_TRY(cudaGetDevice(&dev));
  CHEM_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  // the kernels' limit, and their attribute whatever a launch takes: it is state of the function, and
  // another thread may launch one of another size meanwhile
  constexpr size_t kSmem = 200 * 1024;
  if (ns <= 15) {
    // Whole warps per sub-partition, 4 to 16 an SM as far as shared memory goes, more of them overlap one
    // warp's integer work with the others' FP64 (100003 H2 cells: a pass of the grid takes 43, 49 and
    // 80 us with up to 4, 8 and 16), but the last pass may be nearly empty: the number with the least
    // passes times their length, max(11, warps + 4) units of 4 us.  The units are those of 9 species; with
    // 12 and 15 the rule gives 2.5 to 3 times the rate of four lanes a cell in FP64 from 30011 cells on, and
    // 0.90 to 0.99 of it for about 1000 cells (12 species, mu alone: 43.6 us against 39.5), which use one
    // sub-partition of 32 SMs.
    const size_t fixed = (256 + 8 * (size_t)ns + 4 * npair + 3 * (size_t)ns * ns + ns + (ns & 1)) * 8;
    const size_t per = (size_t)5 * ns * 256;
    const int64_t need = (ncells + 31) / 32;
    const int64_t fit = std::max<int64_t>(1, (int64_t)((kSmem - fixed) / per));
    int64_t best = std::numeric_limits<int64_t>::max();
    int warps = 1;
    for (int64_t w : {16, 12, 8, 4}) {
      w = std::min<int64_t>({w, fit, (need + sms - 1) / sms});
      const int64_t cost = ((need + sms * w - 1) / (sms * w)) * std::max<int64_t>(11, w + 4);
      if (cost < best) { best = cost; warps = (int)w; }
    }
    const size_t smem = fixed + per * warps;
    CHEM_CUDA_TRY(cudaFuncSetAttribute(transport_cell_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmem));
    const unsigned grid = (unsigned)std::min<int64_t>((need + warps - 1) / warps, sms);
    transport_cell_kernel<<<grid, 32 * warps, smem, (cudaStream_t)stream>>>(P);
  } else {
    const size_t smem = (256 + 8 * (size_t)(4 * ns + npair)) * sizeof(double);
    if (smem > kSmem) { set_error("mechanism too large for the transport kernel"); return CHEM_EINVAL; }
    CHEM_CUDA_TRY(cudaFuncSetAttribute(transport_warp_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmem));
    transport_warp_kernel<<<grid_cells(ncells, 8), 256, smem, (cudaStream_t)stream>>>(P);
  }
  CHEM_CUDA_TRY(cudaGetLastError());
  return CHEM_OK;
}
