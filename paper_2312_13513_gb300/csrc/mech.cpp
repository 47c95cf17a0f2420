// Mechanism loading: text parser, validation, device blob and Jacobian-assembly program.
//
// The kinetics model is the one §2 of the paper delegates to Cantera: NASA-7 species thermo
// with two ranges split at 1000 K, modified-Arrhenius rate constants, third-body collision
// partners with per-species efficiencies, Troe fall-off, and reverse rates from equilibrium
// constants.  This file precomputes everything that does not depend on the state (scaled
// polynomial coefficients, Ta = Ea/Rc, ln A, sparse efficiency lists, species production lists)
// into one blob that every CTA stages into shared memory once.
#include <algorithm>
#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <cstring>
#include <fstream>
#include <map>
#include <mutex>
#include <sstream>
#include <string>
#include <vector>

#include <cuda.h>

#include "chem_internal.h"
#include "exp_table.h"
#include "fixed.cuh"

namespace chem {

static thread_local std::string g_err;

void set_error(const char* fmt, ...) {
  char buf[1024];
  va_list ap;
  va_start(ap, fmt);
  vsnprintf(buf, sizeof buf, fmt, ap);
  va_end(ap);
  g_err = buf;
}

int cuda_fail(cudaError_t e, const char* what) {
  set_error("CUDA error in %s: %s", what, cudaGetErrorString(e));
  return e == cudaErrorMemoryAllocation ? CHEM_ENOMEM : CHEM_ECUDA;
}

namespace {

// Memory pools of the library's per-call temporaries, one per device (and context of it).  The default
// pool gives its memory back to the system at every synchronisation, so a caller that waits for each step
// paid the physical allocation again on each call (0.2 ms for a small surrogate step, 4 ms for a
// per-species pass); these pools keep up to kKeepBytes, and give it back when the context's last mechanism
// and model are freed (in that context).  The pools are the driver's own, safe for any number of threads
// and streams.  A context that is gone (a reset device) has taken its pool along: the slot's number is
// never met again, and the handle never used.
constexpr uint64_t kKeepBytes = 512ull << 20;
struct PoolSlot {
  int device = -1;                     // -1: free
  unsigned long long context = 0;
  cudaMemPool_t pool = nullptr;        // null: none could be made
  int users = 0;
};
struct Pools {
  std::mutex mu;
  PoolSlot slot[64];
};
Pools& pools() {
  static Pools* p = new Pools();       // never destroyed: calls may come during process exit
  return *p;
}

// Number of the current device's context, another one after each reset; 0 where there is none.  (Driver
// entry points by the runtime's query: the library does not link the driver library.)
unsigned long long context_number(int dev) {
  typedef CUresult (*CurrentFn)(CUcontext*);
  typedef CUresult (*IdFn)(CUcontext, unsigned long long*);
  struct Fns {
    CurrentFn current = nullptr;
    IdFn id = nullptr;
    Fns() {
      void* p = nullptr;
      cudaDriverEntryPointQueryResult q;
      if (cudaGetDriverEntryPointByVersion("cuCtxGetCurrent", &p, 12000, cudaEnableDefault, &q) == cudaSuccess &&
          q == cudaDriverEntryPointSuccess)
        current = (CurrentFn)p;
      if (cudaGetDriverEntryPointByVersion("cuCtxGetId", &p, 12000, cudaEnableDefault, &q) == cudaSuccess &&
          q == cudaDriverEntryPointSuccess)
        id = (IdFn)p;
    }
  };
  static const Fns f;
  CUcontext c = nullptr;
  unsigned long long n = 0;
  if (!f.current || !f.id) return 0;
  if (f.current(&c) != CUDA_SUCCESS || !c) {         // a host thread's first call binds it here
    if (cudaSetDevice(dev) != cudaSuccess || f.current(&c) != CUDA_SUCCESS || !c) return 0;
  }
  return f.id(c, &n) == CUDA_SUCCESS ? n : 0;
}

// the slot of the current device and context, made with its pool where there is none (under the lock)
PoolSlot* pool_slot(Pools& P, int dev) {
  const unsigned long long c = context_number(dev);
  PoolSlot* empty = nullptr;
  for (PoolSlot& s : P.slot) {
    if (s.device == dev && s.context == c) return &s;
    if (s.device < 0 && !empty) empty = &s;
  }
  if (!empty) return nullptr;
  *empty = PoolSlot{dev, c};
  cudaMemPoolProps props{};
  props.allocType = cudaMemAllocationTypePinned;
  props.location.type = cudaMemLocationTypeDevice;
  props.location.id = dev;
  uint64_t keep = kKeepBytes;
  if (cudaMemPoolCreate(&empty->pool, &props) == cudaSuccess) {
    cudaMemPoolSetAttribute(empty->pool, cudaMemPoolAttrReleaseThreshold, &keep);
  } else {
    empty->pool = nullptr;
    cudaGetLastError();
  }
  return empty;
}

cudaMemPool_t device_pool() {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return nullptr;
  Pools& P = pools();
  std::lock_guard<std::mutex> lk(P.mu);
  const PoolSlot* s = pool_slot(P, dev);
  return s ? s->pool : nullptr;
}

int align16(int x) { return (x + 15) & ~15; }

struct Builder {
  std::vector<unsigned char> buf;
  int add(int bytes) {
    int off = (int)buf.size();
    buf.resize(off + align16(bytes), 0);
    return off;
  }
  template <class T> T* at(int off) { return reinterpret_cast<T*>(buf.data() + off); }
};

// Copy of a mechanism description whose reactions are reordered fall-off first, then
// third-body, then elementary (stable within each class).  The rate loop hands consecutive
// reactions to consecutive threads, so the long fall-off branch runs in as few warps as possible.
struct Reordered {
  chem_mech_desc d{};
  std::vector<int> rtype, reac, prod, has_t2;
  std::vector<double> A, b, Ea, troe, eff;
};

void reorder_reactions(const chem_mech_desc* in, Reordered* o) {
  const int ns = in->n_species, nr = in->n_reactions;
  std::vector<int> order;
  for (int cls : {2, 1, 0})
    for (int j = 0; j < nr; ++j)
      if (in->rtype[j] == cls) order.push_back(j);
  o->d = *in;
  o->rtype.resize(nr); o->reac.resize(3 * nr); o->prod.resize(3 * nr); o->has_t2.resize(nr);
  o->A.resize(nr); o->b.resize(nr); o->Ea.resize(nr); o->troe.resize(7 * (size_t)nr);
  o->eff.resize((size_t)nr * ns);
  for (int jn = 0; jn < nr; ++jn) {
    const int j = order[jn];
    o->rtype[jn] = in->rtype[j];
    for (int i = 0; i < 3; ++i) { o->reac[3 * jn + i] = in->reac[3 * j + i]; o->prod[3 * jn + i] = in->prod[3 * j + i]; }
    o->has_t2[jn] = in->has_t2[j];
    o->A[jn] = in->A[j]; o->b[jn] = in->b[j]; o->Ea[jn] = in->Ea[j];
    for (int i = 0; i < 7; ++i) o->troe[7 * (size_t)jn + i] = in->troe[7 * (size_t)j + i];
    for (int k = 0; k < ns; ++k) o->eff[(size_t)jn * ns + k] = in->eff[(size_t)j * ns + k];
  }
  if (nr > 0) {
    o->d.rtype = o->rtype.data(); o->d.reac = o->reac.data(); o->d.prod = o->prod.data();
    o->d.has_t2 = o->has_t2.data(); o->d.A = o->A.data(); o->d.b = o->b.data(); o->d.Ea = o->Ea.data();
    o->d.troe = o->troe.data(); o->d.eff = o->eff.data();
  }
}

const fx::u64 kExp2Tab[256] = {CHEM_FX_EXP2_VALUES};
const fx::u64 kLog2Tab[128] = {CHEM_FX_LOG2_VALUES};
const uint32_t kRcpTab[128] = {CHEM_FX_RCP_VALUES};

// The numbers of a mechanism in the fixed-point formats (fixed.cuh, fx_mech.h).  ok = false where a
// species' polynomials leave them.  No polynomial can leave Q11.52 (its coefficients' magnitudes
// sum to at most 2000), and every base-2 exponent that a kernel forms stays below 3074 in magnitude
// (|log2 kf| <= 600 + 32 * 12 + 1900; |log2 kr| <= 1023 + 2000 by the bound on Delta G;
// |log2 k0 / kinf| <= 2050 + 1023, of a kinf in range, by a bound on k0 of its own), so that a wrapped
// sum is always recognised as out of range (exp2_in_range) and never mistaken for a small one.
struct FxNumbers {
  bool ok = true;
  std::vector<FxSpecies> sp;                       // [2][ns]
  std::vector<int64_t> lnA;                        // [nr]; 2000 where a reaction is left to FP64
  std::vector<uint64_t> beta, Ta;
  std::vector<FxTroe> troe;
  int64_t lpr0 = 0;
  const long double l2 = std::log(2.0L);
  bool hok = true;                                 // the enthalpy polynomials below fit
  std::vector<FxEnthalpy> hk;                      // [2][ns]

  int64_t q52l(long double v, double lim) {
    if (!(std::fabs((double)v) <= lim)) { ok = false; return 0; }
    return (int64_t)std::nearbyintl(v * 4503599627370496.0L);
  }
  int64_t q56(double v) { return (int64_t)std::nearbyintl((long double)v * 72057594037927936.0L); }

  // |Delta G / (RT ln 2)| of a reaction over [kTlo, kThi): on 128 log-spaced pieces, the value at
  // the left end plus the change of every (monotone) term across the piece
  static double worst_dG(const chem_mech_desc* d, const std::vector<int>& nu, int dnu) {
    const int ns = d->n_species;
    double c[2][7] = {};
    for (int k = 0; k < ns; ++k)
      if (nu[k])
        for (int t = 0; t < 7; ++t) {
          c[0][t] += nu[k] * d->nasa_lo[7 * k + t];
          c[1][t] += nu[k] * d->nasa_hi[7 * k + t];
        }
    double worst = 0.0;
    const double step = std::pow(fx::kThi / fx::kTlo, 1.0 / 128.0);
    double T = fx::kTlo;
    for (int i = 0; i < 128; ++i, T *= step) {
      const double T1 = T * step;
      for (int r = T >= TMID ? 1 : 0; r <= (T1 < TMID ? 0 : 1); ++r) {
        auto terms = [&](double x, double* o) {
          double p = 1.0;
          for (int t = 0; t < 5; ++t, p *= x)
            o[t] = t == 0 ? c[r][0] * (1.0 - std::log(x)) - c[r][6] : -c[r][t] * p / (t * (t + 1));
          o[5] = c[r][5] / x;
          o[6] = dnu * (std::log(x) - std::log(PATM / RU));
        };
        double a0[7], a1[7], v = 0.0, w = 0.0;
        terms(T, a0);
        terms(T1, a1);
        for (int t = 0; t < 7; ++t) { v += a0[t]; w += std::fabs(a1[t] - a0[t]); }
        worst = std::max(worst, std::fabs(v) + w);
      }
    }
    return worst / std::log(2.0);
  }

  static bool in_formats(double A, double b, double Ea) {
    return A > 0.0 && std::fabs(std::log2(A)) <= 599.0 && std::fabs(b) <= 32.0 && std::fabs(Ea / RC) <= 160000.0;
  }
  void rate(double A, double b, double Ea, bool fits, int64_t* lnA_, uint64_t* beta_, uint64_t* Ta_) {
    fits = fits && in_formats(A, b, Ea);
    *lnA_ = fits ? q52l(std::log((long double)A) / l2, 600.0) : (int64_t)2000 << 52;
    *beta_ = fx::biased(fits ? q56(b) : 0);
    *Ta_ = fx::biased(fits ? q52l((long double)Ea / (long double)RC / l2 / 128.0L, 1900.0) : 0);
  }

  FxNumbers(const chem_mech_desc* d, const std::vector<std::vector<int>>& nu, const std::vector<double>& W) {
    const int ns = d->n_species, nr = d->n_reactions;
    sp.resize(2 * (size_t)ns);
    for (int r = 0; r < 2; ++r)
      for (int k = 0; k < ns; ++k) {
        const double* a = (r == 0 ? d->nasa_lo : d->nasa_hi) + 7 * k;
        FxSpecies& S = sp[(size_t)r * ns + k];
        const int sh = r == 0 ? kFxR0 : kFxR1;
        long double p = 1.0L;
        for (int i = 0; i < 5; ++i, p *= std::ldexp(1.0L, sh)) {
          // i-th coefficients of h/RT, s/R (the constant is a7, the T-free part of a1 (1 - ln T) is
          // a1) and cp/R in powers of tau
          S.c[i] = q52l((long double)a[i] * p, 500.0);
          S.h[i] = q52l((long double)a[i] / (i + 1) * p, 500.0);
          const long double s = i == 0 ? (long double)a[6] : (long double)a[i] / i * p;
          const long double g = (i == 0 ? (long double)a[0] : (long double)a[i] / (i + 1) * p) - s;
          S.g[i] = q52l(g / l2, 1000.0);
        }
        S.ha6 = q52l((long double)a[5] / 128.0L, 1900.0);
        S.ga6 = q52l((long double)a[5] / 128.0L / l2, 1900.0);
        if (!(std::fabs(a[0]) <= 100.0)) ok = false;
        S.gl = ok ? q56(-a[0]) : 0;
        double sg = std::fabs((double)S.ga6), sh_ = std::fabs((double)S.ha6), sc = 0.0;
        for (int i = 0; i < 5; ++i) {
          sg += std::fabs((double)S.g[i]); sh_ += std::fabs((double)S.h[i]);
          sc += std::max(1, i) * std::fabs((double)S.c[i]);
        }
        sg += 12.0 * std::fabs((double)S.gl) / 16.0;
        if (!(std::max(std::max(sg, sh_), sc) <= 2000.0 * 4503599627370496.0)) ok = false;
        for (int64_t* x : {&S.g[4], &S.h[4], &S.c[4], &S.ga6, &S.gl, &S.ha6}) *x = (int64_t)fx::biased(*x);
      }
    hk.resize(2 * (size_t)ns);
    for (int r = 0; r < 2; ++r)
      for (int k = 0; k < ns; ++k) {
        const double* a = (r == 0 ? d->nasa_lo : d->nasa_hi) + 7 * k;
        FxEnthalpy& E = hk[(size_t)r * ns + k];
        const long double t = std::ldexp(1.0L, r == 0 ? kFxR0 : kFxR1), w = W[k];
        long double hv[6], cv[5], pw = 1.0L, hs = 0.0L, cs = 0.0L;
        hv[0] = a[5] / w;
        for (int i = 0; i < 5; ++i) {
          cv[i] = a[i] * pw / w;
          pw *= t;
          hv[i + 1] = a[i] / (i + 1) * pw / w;
        }
        for (int i = 0; i < 6; ++i) hs += std::fabs(hv[i]);
        for (int i = 0; i < 5; ++i) cs += std::fabs(cv[i]);
        if (!(hs < 1e12L && cs < 1e12L)) { hok = false; continue; }
        auto frac = [](long double sum) { return sum > 0.0L ? std::min(60, 61 - (int)std::floor(std::log2(sum))) : 60; };
        E.fh = frac(hs * 1.0001L);
        E.fc = frac(cs * 1.0001L);
        for (int i = 0; i < 6; ++i) E.h[i] = (int64_t)std::nearbyintl(std::ldexp(hv[i], E.fh));
        for (int i = 0; i < 5; ++i) E.c[i] = (int64_t)std::nearbyintl(std::ldexp(cv[i], E.fc));
        E.h[5] = (int64_t)fx::biased(E.h[5]);
        E.c[4] = (int64_t)fx::biased(E.c[4]);
        for (int i = 0; i < 5; ++i) E.cf[i] = (float)cv[i];
      }
    lpr0 = q52l(std::log((long double)PATM / (long double)RU) / l2, 1000.0);
    lnA.resize(nr); beta.resize(nr); Ta.resize(nr);
    for (int j = 0; j < nr; ++j) {
      int dnu = 0;
      for (int k = 0; k < ns; ++k) dnu += nu[j][k];
      bool fits = worst_dG(d, nu[j], dnu) <= 2000.0;
      if (d->rtype[j] == 2) {
        const double* t = d->troe + 7 * j;
        fits = fits && in_formats(t[0], t[1], t[2]) &&
               std::fabs(std::log2(t[0])) + 12.0 * std::fabs(t[1]) + std::fabs(t[2]) / (RC * std::log(2.0) * fx::kTlo) <= 2050.0;
        FxTroe F{};
        rate(t[0], t[1], t[2], fits, &F.lnA0, &F.b0, &F.Ta0);
        F.b0d = t[1]; F.Ta0K = t[2] / RC;
        F.a = t[3]; F.iT3 = 1.0 / t[4]; F.iT1 = 1.0 / t[5]; F.T2 = t[6];
        F.has_t2 = d->has_t2[j] ? 1.0 : 0.0;
        troe.push_back(F);
      }
      rate(d->A[j], d->b[j], d->Ea[j], fits, &lnA[j], &beta[j], &Ta[j]);
    }
  }
};

// third-body sets in reaction order: sparse (efficiency - 1) and, dense, the efficiencies
struct Partners {
  std::vector<int> off{0};
  std::vector<int16_t> idx;
  std::vector<double> val, dense;
  std::vector<int16_t> tb_of, troe_of;
  int ntb = 0, ntroe = 0;
  explicit Partners(const chem_mech_desc* d) : tb_of(d->n_reactions, -1), troe_of(d->n_reactions, -1) {
    const int ns = d->n_species;
    for (int j = 0; j < d->n_reactions; ++j) {
      if (d->rtype[j] == 0) continue;
      tb_of[j] = (int16_t)ntb++;
      if (d->rtype[j] == 2) troe_of[j] = (int16_t)ntroe++;
      for (int k = 0; k < ns; ++k) {
        const double e = d->eff[(size_t)j * ns + k];
        dense.push_back(e);
        if (e != 1.0) { idx.push_back((int16_t)k); val.push_back(e - 1.0); }
      }
      off.push_back((int)idx.size());
    }
  }
};

template <class T>
void put(Builder& B, int off, const std::vector<T>& v) {
  if (!v.empty()) memcpy(B.at<unsigned char>(off), v.data(), v.size() * sizeof(T));
}

// Blob of the cell-per-thread kernel (fx_mech.h); L->bytes = 0 where there is none.
std::vector<unsigned char> build_fx(const chem_mech_desc* d, const chem_mech_s* m, const FxNumbers& F,
                                    const std::vector<std::vector<int>>& nu, FxLayout* L) {
  const int ns = d->n_species, nr = d->n_reactions;
  *L = FxLayout{};
  if (!F.ok || ns < kCellMinNs || ns > kCellMaxNs || nr > 1024) return {};
  const Partners T(d);
  Builder B;
  L->ns = ns; L->ntb = T.ntb; L->lpr0 = F.lpr0;
  // at most two species per side and four net species: FxRate, by type; the rest: FxReac
  std::vector<int> order[4];
  for (int j = 0; j < nr; ++j) {
    int nre = 0, npr = 0, nn = 0;
    for (int i = 0; i < 3; ++i) { nre += d->reac[3 * j + i] >= 0; npr += d->prod[3 * j + i] >= 0; }
    for (int k = 0; k < ns; ++k) nn += nu[j][k] != 0;
    order[nre <= 2 && npr <= 2 && nn <= 4 ? d->rtype[j] : 3].push_back(j);
  }
  L->n_plain = (int)order[0].size(); L->n_tb = (int)order[1].size(); L->n_fo = (int)order[2].size();
  L->n_gen = (int)order[3].size();
  L->o_exp2 = B.add(sizeof(kExp2Tab));
  L->o_lg = B.add(sizeof(kLog2Tab));
  L->o_rcp = B.add(sizeof(kRcpTab));
  L->o_sp = B.add(2 * ns * (int)sizeof(FxSpecies));
  L->o_W = B.add(8 * ns);
  L->o_invW = B.add(8 * ns);
  L->o_nu = B.add(8 * 16);
  L->o_rate = B.add((nr - L->n_gen) * (int)sizeof(FxRate));
  L->o_reac = B.add(L->n_gen * (int)sizeof(FxReac));
  L->o_troe = B.add(T.ntroe * (int)sizeof(FxTroe));
  L->o_effv = B.add(8 * (int)T.val.size());
  L->o_eff = B.add(8 * (int)T.dense.size());
  L->o_effidx = B.add(2 * (int)T.idx.size());
  L->o_effoff = B.add(4 * (int)T.off.size());
  memcpy(B.at<unsigned char>(L->o_exp2), kExp2Tab, sizeof(kExp2Tab));
  memcpy(B.at<unsigned char>(L->o_lg), kLog2Tab, sizeof(kLog2Tab));
  memcpy(B.at<unsigned char>(L->o_rcp), kRcpTab, sizeof(kRcpTab));
  put(B, L->o_sp, F.sp); put(B, L->o_troe, F.troe); put(B, L->o_effv, T.val); put(B, L->o_eff, T.dense);
  put(B, L->o_effidx, T.idx); put(B, L->o_effoff, T.off);
  for (int k = 0; k < ns; ++k) {
    B.at<double>(L->o_W)[k] = m->W[k];
    B.at<double>(L->o_invW)[k] = 1.0 / m->W[k];
  }
  for (int c = 0; c < 16; ++c) B.at<double>(L->o_nu)[c] = (double)(c - 8);
  FxRate* R = B.at<FxRate>(L->o_rate);
  for (int cls = 0; cls < 3; ++cls)
    for (int j : order[cls]) {
      int dnu = 0, nr_ = 0, np_ = 2;
      for (int i = 0; i < 4; ++i) R->c[i] = (uint16_t)(ns * 256);
      for (int i = 0; i < 3; ++i) {
        if (d->reac[3 * j + i] >= 0) { R->c[nr_++] = (uint16_t)(d->reac[3 * j + i] * 256); --dnu; }
        if (d->prod[3 * j + i] >= 0) { R->c[np_++] = (uint16_t)(d->prod[3 * j + i] * 256); ++dnu; }
      }
      R->dnu = (int16_t)dnu; R->id = (int16_t)j; R->tb = T.tb_of[j]; R->troe = T.troe_of[j];
      R->lnA = F.lnA[j]; R->beta = F.beta[j]; R->Ta = F.Ta[j];
      R->b = d->b[j];
      R->TaK = d->Ea[j] / RC;
      int n = 0;
      for (int pass = 0; pass < 2; ++pass)                      // net species first, then fillers
        for (int k = 0; k < ns && n < 4; ++k)
          if ((nu[j][k] != 0) == (pass == 0)) { R->w[n] = (uint16_t)(k * 256); R->nu[n++] = nu[j][k]; }
      ++R;
    }
  FxReac* G = B.at<FxReac>(L->o_reac);
  for (int j : order[3]) {
    int dnu = 0;
    for (int i = 0; i < 3; ++i) {
      if (d->reac[3 * j + i] >= 0) { G->re[G->nre++] = (uint8_t)d->reac[3 * j + i]; --dnu; }
      if (d->prod[3 * j + i] >= 0) { G->pr[G->npr++] = (uint8_t)d->prod[3 * j + i]; ++dnu; }
    }
    G->dnu = (int16_t)dnu; G->id = (int16_t)j; G->tb = T.tb_of[j]; G->troe = T.troe_of[j];
    G->type = (uint8_t)d->rtype[j];
    G->lnA = F.lnA[j]; G->beta = F.beta[j]; G->Ta = F.Ta[j];
    G->b = d->b[j];
    G->TaK = d->Ea[j] / RC;
    for (int k = 0; k < ns; ++k)
      if (nu[j][k] != 0) { G->sp[G->nnet] = (uint8_t)k; G->nu[G->nnet++] = (int8_t)nu[j][k]; }
    ++G;
  }
  L->bytes = (int)B.buf.size();
  return B.buf;
}

// gather programs of the blob that build_fx made (CoLayout)
std::vector<unsigned char> build_co(const std::vector<unsigned char>& fxb, const FxLayout& F, CoLayout* L) {
  *L = CoLayout{};
  if (!F.bytes || F.n_gen) return {};
  const int ns = F.ns, N = ns + 1, n = F.n_plain + F.n_tb + F.n_fo;
  const FxRate* R = (const FxRate*)(fxb.data() + F.o_rate);
  const double* eff = (const double*)(fxb.data() + F.o_eff);
  std::vector<std::vector<int>> wt(ns);
  std::vector<std::vector<CoTerm>> en((size_t)ns * ns);
  for (int j = 0; j < n; ++j) {
    for (int i = 0; i < 4; ++i)
      if (R[j].nu[i] != 0.0) wt[R[j].w[i] / 256].push_back(j << 4 | ((int)R[j].nu[i] + 8));
    for (int s = 0; s < 4; ++s) {
      if (R[j].c[s] / 256 == ns) continue;
      for (int i = 0; i < 4; ++i)
        if (R[j].nu[i] != 0.0) en[(size_t)(R[j].w[i] / 256) * ns + R[j].c[s] / 256].push_back({-R[j].nu[i], 4 * j + s, 0});
    }
    if (j < F.n_plain) continue;
    for (int i = 0; i < 4; ++i)
      if (R[j].nu[i] != 0.0)
        for (int k = 0; k < ns; ++k)
          en[(size_t)(R[j].w[i] / 256) * ns + k].push_back({-R[j].nu[i] * eff[R[j].tb * ns + k], 4 * n + j - F.n_plain, 0});
  }
  std::vector<int> order, woff(1, 0), wterm, eoff(1, 0), epos;
  std::vector<CoTerm> term;
  for (int k = 0; k < ns; ++k) { wterm.insert(wterm.end(), wt[k].begin(), wt[k].end()); woff.push_back((int)wterm.size()); }
  for (int e = 0; e < ns * ns; ++e)
    if (!en[e].empty()) order.push_back(e);
  std::stable_sort(order.begin(), order.end(), [&](int a, int b) { return en[a].size() > en[b].size(); });
  for (int e : order) {
    term.insert(term.end(), en[e].begin(), en[e].end());
    eoff.push_back((int)term.size());
    epos.push_back((1 + e / ns) * N + 1 + e % ns);
  }
  Builder B;
  L->n = n; L->nent = (int)order.size(); L->nval = 4 * n + F.n_tb + F.n_fo;
  L->o_woff = B.add(4 * (int)woff.size());
  L->o_wterm = B.add(4 * (int)wterm.size());
  L->o_eoff = B.add(4 * (int)eoff.size());
  L->o_epos = B.add(4 * (int)epos.size());
  L->o_term = B.add((int)(sizeof(CoTerm) * term.size()));
  put(B, L->o_woff, woff); put(B, L->o_wterm, wterm); put(B, L->o_eoff, eoff); put(B, L->o_epos, epos);
  put(B, L->o_term, term);
  L->bytes = (int)B.buf.size();
  return B.buf;
}

// Blob of the group kernels' fixed-point form, and their Jacobian program (one global allocation
// each, uploaded here).
int build_gx(const chem_mech_desc* d, chem_mech_s* m, const FxNumbers& F, const std::vector<std::vector<int>>& nu,
             const MechLayout& ML, const Builder& MB) {
  const int ns = d->n_species, nr = d->n_reactions;
  m->gx = GxLayout{};
  if (!F.ok) return CHEM_OK;
  const Partners T(d);
  GxLayout L{};
  Builder B;
  L.ns = ns; L.nr = nr; L.ntb = T.ntb; L.npieces = ML.npieces; L.lpr0 = F.lpr0;
  L.o_exp2 = B.add(sizeof(kExp2Tab));
  L.o_sp = B.add(2 * ns * (int)sizeof(FxSpecies));
  L.o_W = B.add(8 * ns);
  L.o_invW = B.add(8 * ns);
  L.o_nu = B.add(8 * 16);
  L.o_lnA = B.add(8 * nr);
  L.o_beta = B.add(8 * nr);
  L.o_Ta = B.add(8 * nr);
  L.o_reac = B.add(8 * nr);
  L.o_prod = B.add(8 * nr);
  L.o_rinfo = B.add(8 * nr);
  L.o_troe = B.add(T.ntroe * (int)sizeof(FxTroe));
  L.o_effv = B.add(8 * (int)T.val.size());
  L.o_effidx = B.add(2 * (int)T.idx.size());
  L.o_effoff = B.add(4 * (int)T.off.size());
  const int np = ML.nprod;
  L.o_wpk = B.add(4 * np);
  L.o_pterm = B.add(4 * (ML.npieces + 1));
  L.o_poff = B.add(4 * (ns + 1));
  memcpy(B.at<unsigned char>(L.o_exp2), kExp2Tab, sizeof(kExp2Tab));
  put(B, L.o_sp, F.sp); put(B, L.o_lnA, F.lnA); put(B, L.o_beta, F.beta); put(B, L.o_Ta, F.Ta);
  put(B, L.o_troe, F.troe); put(B, L.o_effv, T.val); put(B, L.o_effidx, T.idx); put(B, L.o_effoff, T.off);
  memcpy(B.at<unsigned char>(L.o_W), MB.buf.data() + ML.o_W, 8 * ns);
  memcpy(B.at<unsigned char>(L.o_invW), MB.buf.data() + ML.o_invW, 8 * ns);
  for (int c = 0; c < 16; ++c) B.at<double>(L.o_nu)[c] = (double)(c - 8);
  memcpy(B.at<unsigned char>(L.o_reac), MB.buf.data() + ML.o_reac, 8 * (size_t)nr);
  memcpy(B.at<unsigned char>(L.o_prod), MB.buf.data() + ML.o_prod, 8 * (size_t)nr);
  memcpy(B.at<unsigned char>(L.o_rinfo), MB.buf.data() + ML.o_rinfo, 8 * (size_t)nr);
  for (int e = 0; e < 4 * nr; ++e) {
    int16_t* r = B.at<int16_t>(L.o_reac) + e;
    int16_t* p = B.at<int16_t>(L.o_prod) + e;
    if (*r < 0) *r = (int16_t)ns;
    if (*p < 0) *p = (int16_t)ns;
  }
  memcpy(B.at<unsigned char>(L.o_wpk), MB.buf.data() + ML.o_wpk, 4 * (size_t)np);
  memcpy(B.at<unsigned char>(L.o_pterm), MB.buf.data() + ML.o_pterm, 4 * (size_t)(ML.npieces + 1));
  memcpy(B.at<unsigned char>(L.o_poff), MB.buf.data() + ML.o_poff, 4 * (size_t)(ns + 1));
  L.bytes = (int)B.buf.size();

  struct Entry {
    std::vector<std::pair<int, int>> slot;       // (src, oth)
    std::vector<std::pair<int, double>> part;    // (set, coef)
  };
  std::map<std::pair<int, int>, Entry> ent;
  std::vector<std::vector<int>> rows(ns);
  for (int j = 0; j < nr; ++j)
    for (int k = 0; k < ns; ++k) {
      if (nu[j][k] == 0) continue;
      for (int s = 0; s < 6; ++s) {
        const int* side = s < 3 ? d->reac + 3 * j : d->prod + 3 * j;
        const int sl = s % 3;
        if (side[sl] < 0) continue;
        const int a1 = sl == 0 ? 1 : 0, a2 = sl == 2 ? 1 : 2;
        const int o1 = side[a1] >= 0 ? side[a1] : ns, o2 = side[a2] >= 0 ? side[a2] : ns;
        for (int u = 0; u < std::abs(nu[j][k]); ++u)
          ent[{k, side[sl]}].slot.push_back({((2 * j + (s >= 3)) << 1) | (nu[j][k] < 0), o1 | (o2 << 16)});
      }
      if (T.tb_of[j] < 0) continue;
      rows[k].push_back((T.tb_of[j] << 4) | (nu[j][k] + 8));
      for (int e = T.off[T.tb_of[j]]; e < T.off[T.tb_of[j] + 1]; ++e)
        ent[{k, T.idx[e]}].part.push_back({T.tb_of[j], nu[j][k] * T.val[e]});
    }
  // entries with many terms first, so that the lanes of a chunk have similar counts
  std::vector<const std::pair<const std::pair<int, int>, Entry>*> order;
  for (auto& kv : ent) order.push_back(&kv);
  std::stable_sort(order.begin(), order.end(), [](const auto* a, const auto* b) {
    if (a->second.slot.size() != b->second.slot.size()) return a->second.slot.size() > b->second.slot.size();
    return a->second.part.size() > b->second.part.size();
  });
  std::vector<int> ro(1, 0), rs;
  std::vector<int4> ss;
  std::vector<int2> pt;
  std::vector<double> pc;
  for (size_t e0 = 0; e0 < order.size(); e0 += kGxLanes) {
    const size_t e1 = std::min(order.size(), e0 + kGxLanes);
    size_t nsl = 1, npt = 0;                         // every entry is written by the slot pass
    for (size_t e = e0; e < e1; ++e) {
      nsl = std::max(nsl, order[e]->second.slot.size());
      npt = std::max(npt, order[e]->second.part.size());
    }
    const size_t s0 = ss.size(), p0 = pt.size();
    ss.resize(s0 + nsl * kGxLanes, int4{(2 * nr) << 1, ns | (ns << 16), -1, 0});
    pt.resize(p0 + npt * kGxLanes, int2{0, -1});
    pc.resize(p0 + npt * kGxLanes, 0.0);
    for (size_t e = e0; e < e1; ++e) {
      const Entry& E = order[e]->second;
      const int pos = (order[e]->first.first << 16) | order[e]->first.second;
      for (size_t i = 0; i < E.slot.size(); ++i) {
        int4& t = ss[s0 + i * kGxLanes + (e - e0)];
        t.x = E.slot[i].first;
        t.y = E.slot[i].second;
      }
      ss[s0 + (nsl - 1) * kGxLanes + (e - e0)].z = pos;
      for (size_t i = 0; i < E.part.size(); ++i) {
        pt[p0 + i * kGxLanes + (e - e0)].x = E.part[i].first;
        pc[p0 + i * kGxLanes + (e - e0)] = E.part[i].second;
      }
      if (npt && !E.part.empty()) pt[p0 + (npt - 1) * kGxLanes + (e - e0)].y = pos;
    }
  }
  // whole units of rows, and at least one of slots, which the kernel reads ahead unconditionally (no
  // entries: no reactions, or none with a net production)
  const size_t unit = (size_t)kGxLanes * kGxUnroll;
  ss.resize(std::max<size_t>(1, (ss.size() + unit - 1) / unit) * unit, int4{(2 * nr) << 1, ns | (ns << 16), -1, 0});
  pt.resize((pt.size() + unit - 1) / unit * unit, int2{0, -1});
  pc.resize(pt.size(), 0.0);
  for (int k = 0; k < ns; ++k) { rs.insert(rs.end(), rows[k].begin(), rows[k].end()); ro.push_back((int)rs.size()); }
  Builder J;
  const int o_ss = J.add(16 * (int)ss.size()), o_pt = J.add(8 * (int)pt.size()), o_pc = J.add(8 * (int)pc.size()),
            o_ro = J.add(4 * (int)ro.size()), o_rs = J.add(4 * (int)rs.size());
  put(J, o_ss, ss); put(J, o_pt, pt); put(J, o_pc, pc); put(J, o_ro, ro); put(J, o_rs, rs);
  CHEM_CUDA_TRY(cudaMalloc(&m->d_gx, B.buf.size()));
  CHEM_CUDA_TRY(cudaMemcpy(m->d_gx, B.buf.data(), B.buf.size(), cudaMemcpyHostToDevice));
  CHEM_CUDA_TRY(cudaMalloc(&m->d_gxj, J.buf.size()));
  CHEM_CUDA_TRY(cudaMemcpy(m->d_gxj, J.buf.data(), J.buf.size(), cudaMemcpyHostToDevice));
  const unsigned char* g = (const unsigned char*)m->d_gxj;
  m->gxj = GxJac{(int)(ss.size() / kGxLanes), (int)(pt.size() / kGxLanes), (const int4*)(g + o_ss),
                 (const int2*)(g + o_pt),     (const double*)(g + o_pc),   (const int*)(g + o_ro),
                 (const int*)(g + o_rs)};
  m->gx = L;
  return CHEM_OK;
}

int build(const chem_mech_desc* din, chem_mech_s* m) {
  Reordered ro;
  reorder_reactions(din, &ro);
  const chem_mech_desc* d = &ro.d;
  const int ns = d->n_species, ne = d->n_elements, nr = d->n_reactions;
  m->ns = ns; m->ne = ne; m->nr = nr;
  m->elem_mass.assign(d->elem_mass, d->elem_mass + ne);
  m->comp.assign(d->comp, d->comp + (size_t)ns * ne);
  m->W.assign(ns, 0.0);
  for (int k = 0; k < ns; ++k)
    for (int e = 0; e < ne; ++e) m->W[k] += d->comp[(size_t)k * ne + e] * d->elem_mass[e];
  m->nasa_lo.assign(d->nasa_lo, d->nasa_lo + 7 * ns);
  m->nasa_hi.assign(d->nasa_hi, d->nasa_hi + 7 * ns);

  // third-body sets and troe parameters
  std::vector<int> tb_of(nr, -1), troe_of(nr, -1);
  std::vector<int> eff_off(1, 0);
  std::vector<int16_t> eff_idx;
  std::vector<double> eff_val;
  int ntb = 0, ntroe = 0;
  for (int j = 0; j < nr; ++j) {
    if (d->rtype[j] == 0) continue;
    tb_of[j] = ntb++;
    for (int k = 0; k < ns; ++k) {
      double e = d->eff[(size_t)j * ns + k];
      if (e != 1.0) { eff_idx.push_back((int16_t)k); eff_val.push_back(e - 1.0); }
    }
    eff_off.push_back((int)eff_idx.size());
    if (d->rtype[j] == 2) troe_of[j] = ntroe++;
  }
  // species production lists: (reaction, net stoichiometric coefficient), ascending reaction
  std::vector<std::vector<std::pair<int, int>>> plist(ns);
  std::vector<std::vector<int>> nu(nr, std::vector<int>(ns, 0));
  for (int j = 0; j < nr; ++j) {
    for (int i = 0; i < 3; ++i) {
      if (d->reac[3 * j + i] >= 0) nu[j][d->reac[3 * j + i]] -= 1;
      if (d->prod[3 * j + i] >= 0) nu[j][d->prod[3 * j + i]] += 1;
    }
    for (int k = 0; k < ns; ++k)
      if (nu[j][k] != 0) plist[k].push_back({j, nu[j][k]});
  }
  std::vector<int> woff(ns + 1, 0);
  for (int k = 0; k < ns; ++k) woff[k + 1] = woff[k] + (int)plist[k].size();
  const int nprod = woff[ns];
  // Balanced pieces of the production lists for groups wider than a warp: each species' list
  // is cut into pieces of at most plen terms, plen the smallest that gives at most kPieceTarget
  // pieces, so that one pass of a 128-thread group covers them with similar loop lengths.
  constexpr int kPieceTarget = 128;
  int plen = 1;
  auto count_pieces = [&](int len) {
    int c = 0;
    for (int k = 0; k < ns; ++k) c += std::max(1, ((int)plist[k].size() + len - 1) / len);
    return c;
  };
  while (count_pieces(plen) > kPieceTarget && plen < std::max(1, nprod)) ++plen;
  std::vector<int> pterm(1, 0), poff(ns + 1, 0);
  for (int k = 0; k < ns; ++k) {
    const int len = (int)plist[k].size();
    const int np = std::max(1, (len + plen - 1) / plen);
    for (int i = 0; i < np; ++i) pterm.push_back(woff[k] + std::min(len, (i + 1) * plen));
    poff[k + 1] = poff[k] + np;
  }
  const int npieces = poff[ns];
  const int neff = (int)eff_idx.size();

  MechLayout L{};
  L.ns = ns; L.nr = nr; L.N = ns + 1; L.ntb = ntb; L.ntroe = ntroe; L.nprod = nprod;
  L.npieces = npieces;
  Builder B;
  L.o_W = B.add(8 * ns);
  L.o_invW = B.add(8 * ns);
  L.o_hc = B.add(8 * 2 * ns * 6);
  L.o_sc = B.add(8 * 2 * ns * 6);
  L.o_cpc = B.add(8 * 2 * ns * 5);
  L.o_lnA = B.add(8 * nr);
  L.o_beta = B.add(8 * nr);
  L.o_Ta = B.add(8 * nr);
  L.o_troe = B.add(8 * 8 * ntroe);
  L.o_effv = B.add(8 * neff);
  L.o_const = B.add(8 * kConsts);
  L.o_reac = B.add(2 * 4 * nr);
  L.o_prod = B.add(2 * 4 * nr);
  L.o_rinfo = B.add(2 * 4 * nr);
  L.o_effidx = B.add(2 * neff);
  L.o_wpk = B.add(4 * nprod);
  L.o_effoff = B.add(4 * (ntb + 1));
  L.o_woff = B.add(4 * (ns + 1));
  L.o_pterm = B.add(4 * (npieces + 1));
  L.o_poff = B.add(4 * (ns + 1));
  L.bytes = (int)B.buf.size();

  double* W = B.at<double>(L.o_W);
  double* invW = B.at<double>(L.o_invW);
  for (int k = 0; k < ns; ++k) { W[k] = m->W[k]; invW[k] = 1.0 / m->W[k]; }
  for (int r = 0; r < 2; ++r) {
    const double* src = r == 0 ? d->nasa_lo : d->nasa_hi;
    for (int k = 0; k < ns; ++k) {
      const double* a = src + 7 * k;
      double* hc = B.at<double>(L.o_hc) + (r * ns + k) * 6;
      double* sc = B.at<double>(L.o_sc) + (r * ns + k) * 6;
      double* cc = B.at<double>(L.o_cpc) + (r * ns + k) * 5;
      hc[0] = a[0]; hc[1] = a[1] / 2.0; hc[2] = a[2] / 3.0; hc[3] = a[3] / 4.0; hc[4] = a[4] / 5.0; hc[5] = a[5];
      sc[0] = a[0]; sc[1] = a[1]; sc[2] = a[2] / 2.0; sc[3] = a[3] / 3.0; sc[4] = a[4] / 4.0; sc[5] = a[6];
      for (int i = 0; i < 5; ++i) cc[i] = a[i];
    }
  }
  for (int j = 0; j < nr; ++j) {
    B.at<double>(L.o_lnA)[j] = std::log(d->A[j]);      // A = 0 gives -inf: kf = 0 exactly
    B.at<double>(L.o_beta)[j] = d->b[j];
    B.at<double>(L.o_Ta)[j] = d->Ea[j] / RC;
    int16_t* re = B.at<int16_t>(L.o_reac) + 4 * j;
    int16_t* pr = B.at<int16_t>(L.o_prod) + 4 * j;
    int dnu = 0;
    for (int i = 0; i < 3; ++i) {
      re[i] = (int16_t)d->reac[3 * j + i];
      pr[i] = (int16_t)d->prod[3 * j + i];
      dnu += (d->prod[3 * j + i] >= 0) - (d->reac[3 * j + i] >= 0);
    }
    re[3] = pr[3] = -1;
    int16_t* ri = B.at<int16_t>(L.o_rinfo) + 4 * j;
    ri[0] = (int16_t)d->rtype[j]; ri[1] = (int16_t)dnu; ri[2] = (int16_t)tb_of[j];
    ri[3] = (int16_t)troe_of[j];
    if (troe_of[j] >= 0) {
      const double* t = d->troe + 7 * j;
      double* o = B.at<double>(L.o_troe) + 8 * troe_of[j];
      o[0] = std::log(t[0]); o[1] = t[1]; o[2] = t[2] / RC; o[3] = t[3];
      o[4] = 1.0 / t[4]; o[5] = 1.0 / t[5]; o[6] = t[6]; o[7] = d->has_t2[j] ? 1.0 : 0.0;
    }
  }
  for (int i = 0; i < neff; ++i) {
    B.at<double>(L.o_effv)[i] = eff_val[i];
    B.at<int16_t>(L.o_effidx)[i] = eff_idx[i];
  }
  for (int i = 0; i <= ntb; ++i) B.at<int>(L.o_effoff)[i] = eff_off[i];
  for (int k = 0; k <= ns; ++k) B.at<int>(L.o_woff)[k] = woff[k];
  for (int i = 0; i <= npieces; ++i) B.at<int>(L.o_pterm)[i] = pterm[i];
  for (int k = 0; k <= ns; ++k) B.at<int>(L.o_poff)[k] = poff[k];
  for (int k = 0; k < ns; ++k)
    for (int i = 0; i < (int)plist[k].size(); ++i) {
      const int nuk = plist[k][i].second;
      if (nuk < -8 || nuk > 7) {
        set_error("reaction %d: stoichiometric coefficient %d of species %d out of range", plist[k][i].first, nuk, k);
        return CHEM_EINVAL;
      }
      B.at<int>(L.o_wpk)[woff[k] + i] = (plist[k][i].first << 4) | (nuk + 8);
    }
  double* cst = B.at<double>(L.o_const);
  for (int c = 0; c < 16; ++c) cst[kC_NU + c] = (double)(c - 8);
  cst[kC_LNPR0] = std::log(PATM / RU);
  cst[kC_INVNS] = 1.0 / ns;
  for (int j = 0; j < 64; ++j) cst[kC_EXPTAB + j] = kExpTable[j];
  m->lay = L;

  // Jacobian-assembly program for d(wdot_k)/dC_m; a term is (src, oth, coef)
  struct Term { int src, oth; double coef; };
  std::map<std::pair<int, int>, std::vector<Term>> ent;
  for (int j = 0; j < nr; ++j) {
    for (int k = 0; k < ns; ++k) {
      if (nu[j][k] == 0) continue;
      for (int s = 0; s < 6; ++s) {
        const int* side = s < 3 ? d->reac + 3 * j : d->prod + 3 * j;
        const int sl = s % 3;
        const int sp = side[sl];
        if (sp < 0) continue;
        // the other two slots of the same side, in slot order
        const int a1 = sl == 0 ? 1 : 0, a2 = sl == 2 ? 1 : 2;
        const int o1 = side[a1] >= 0 ? side[a1] : ns, o2 = side[a2] >= 0 ? side[a2] : ns;
        ent[{k, sp}].push_back({(j << 3) | s, o1 | (o2 << 16), (double)nu[j][k]});
      }
      if (d->rtype[j] != 0)
        for (int mm = 0; mm < ns; ++mm) {
          double e = d->eff[(size_t)j * ns + mm];
          if (e != 0.0) ent[{k, mm}].push_back({(j << 3) | 7, 0, nu[j][k] * e});
        }
    }
  }
  JacProgram& P = m->jac;
  P.nent = (int)ent.size();
  std::vector<int> off(1, 0);
  std::vector<int16_t> rows, cols;
  std::vector<int> src, oth;
  std::vector<double> coef;
  // entries with many terms first: threads take consecutive entries, so a warp's entries have
  // similar term counts and its lanes stay busy for the same number of iterations
  std::vector<const std::pair<const std::pair<int, int>, std::vector<Term>>*> order;
  for (auto& kv : ent) order.push_back(&kv);
  std::stable_sort(order.begin(), order.end(),
                   [](const auto* a, const auto* b) { return a->second.size() > b->second.size(); });
  for (auto* kvp : order) {
    const auto& kv = *kvp;
    rows.push_back((int16_t)kv.first.first);
    cols.push_back((int16_t)kv.first.second);
    for (auto& t : kv.second) { src.push_back(t.src); oth.push_back(t.oth); coef.push_back(t.coef); }
    off.push_back((int)src.size());
  }
  P.nterm = (int)src.size();

  const FxNumbers fxn(d, nu, m->W);
  {
    // the tables of fixed.cuh in global memory (step control of every kernel, transport fits) and
    // the enthalpy polynomials (thermo kernels, surrogate post-processing)
    Builder T;
    const int o0 = T.add(sizeof(kExp2Tab)), o1 = T.add(sizeof(kLog2Tab)), o2 = T.add(sizeof(kRcpTab));
    memcpy(T.at<unsigned char>(o0), kExp2Tab, sizeof(kExp2Tab));
    memcpy(T.at<unsigned char>(o1), kLog2Tab, sizeof(kLog2Tab));
    memcpy(T.at<unsigned char>(o2), kRcpTab, sizeof(kRcpTab));
    const int o3 = T.add((int)(fxn.hk.size() * sizeof(FxEnthalpy)));
    put(T, o3, fxn.hk);
    CHEM_CUDA_TRY(cudaMalloc(&m->d_tab, T.buf.size()));
    CHEM_CUDA_TRY(cudaMemcpy(m->d_tab, T.buf.data(), T.buf.size(), cudaMemcpyHostToDevice));
    const unsigned char* t = (const unsigned char*)m->d_tab;
    m->d_e2 = (const unsigned long long*)(t + o0);
    m->d_lg = (const unsigned long long*)(t + o1);
    m->d_rc = (const unsigned int*)(t + o2);
    m->d_hk = fxn.hok ? (const FxEnthalpy*)(t + o3) : nullptr;
  }
  const std::vector<unsigned char> fxb = build_fx(d, m, fxn, nu, &m->fx);
  CHEM_CUDA_TRY(cudaGetDevice(&m->device));
  device_pool();                       // made here: the first call may be under stream capture
  {
    const int rc = build_gx(d, m, fxn, nu, L, B);
    if (rc) return rc;
  }
  if (m->fx.bytes) {
    CHEM_CUDA_TRY(cudaMalloc(&m->d_fx, m->fx.bytes));
    CHEM_CUDA_TRY(cudaMemcpy(m->d_fx, fxb.data(), m->fx.bytes, cudaMemcpyHostToDevice));
    const std::vector<unsigned char> cob = build_co(fxb, m->fx, &m->co);
    if (m->co.bytes) {
      CHEM_CUDA_TRY(cudaMalloc(&m->d_co, m->co.bytes));
      CHEM_CUDA_TRY(cudaMemcpy(m->d_co, cob.data(), m->co.bytes, cudaMemcpyHostToDevice));
    }
  }
  CHEM_CUDA_TRY(cudaMalloc(&m->d_blob, L.bytes));
  CHEM_CUDA_TRY(cudaMemcpy(m->d_blob, B.buf.data(), L.bytes, cudaMemcpyHostToDevice));
  size_t o_off = 0;
  size_t o_row = align16((int)(o_off + 4 * (P.nent + 1)));
  size_t o_col = o_row + align16(2 * P.nent);
  size_t o_src = o_col + align16(2 * P.nent);
  size_t o_oth = o_src + align16(4 * P.nterm);
  size_t o_coef = o_oth + align16(4 * P.nterm);
  size_t tot = o_coef + 8 * (size_t)P.nterm + 16;
  std::vector<unsigned char> jb(tot, 0);
  memcpy(jb.data() + o_off, off.data(), 4 * off.size());
  if (P.nent) {
    memcpy(jb.data() + o_row, rows.data(), 2 * rows.size());
    memcpy(jb.data() + o_col, cols.data(), 2 * cols.size());
  }
  if (P.nterm) {
    memcpy(jb.data() + o_src, src.data(), 4 * src.size());
    memcpy(jb.data() + o_oth, oth.data(), 4 * oth.size());
    memcpy(jb.data() + o_coef, coef.data(), 8 * coef.size());
  }
  CHEM_CUDA_TRY(cudaMalloc(&m->d_jac, tot));
  CHEM_CUDA_TRY(cudaMemcpy(m->d_jac, jb.data(), tot, cudaMemcpyHostToDevice));
  unsigned char* base = (unsigned char*)m->d_jac;
  P.ent_off = (int*)(base + o_off);
  P.ent_row = (int16_t*)(base + o_row);
  P.ent_col = (int16_t*)(base + o_col);
  P.term_src = (int*)(base + o_src);
  P.term_oth = (int*)(base + o_oth);
  P.term_coef = (double*)(base + o_coef);
  return CHEM_OK;
}

int validate(const chem_mech_desc* d) {
  if (!d) { set_error("NULL mechanism description"); return CHEM_EINVAL; }
  const int ns = d->n_species, ne = d->n_elements, nr = d->n_reactions;
  if (ns < 1 || ns > 4096 || ne < 1 || ne > 64 || nr < 0 || nr > 30000) {
    set_error("mechanism sizes out of range (ns=%d ne=%d nr=%d)", ns, ne, nr);
    return CHEM_EINVAL;
  }
  if (!d->elem_mass || !d->comp || !d->nasa_lo || !d->nasa_hi ||
      (nr > 0 && (!d->rtype || !d->reac || !d->prod || !d->A || !d->b || !d->Ea || !d->troe ||
                  !d->has_t2 || !d->eff))) {
    set_error("NULL array in mechanism description");
    return CHEM_EINVAL;
  }
  for (int e = 0; e < ne; ++e)
    if (!(d->elem_mass[e] > 0.0) || !std::isfinite(d->elem_mass[e])) {
      set_error("element %d has a non-positive or non-finite atomic mass", e);
      return CHEM_EINVAL;
    }
  for (int k = 0; k < ns; ++k) {
    double W = 0.0;
    for (int e = 0; e < ne; ++e) {
      if (d->comp[(size_t)k * ne + e] < 0) { set_error("species %d has a negative element count", k); return CHEM_EINVAL; }
      W += d->comp[(size_t)k * ne + e] * d->elem_mass[e];
    }
    if (!(W > 0.0)) { set_error("species %d has non-positive molar mass", k); return CHEM_EINVAL; }
    for (int i = 0; i < 7; ++i)
      if (!std::isfinite(d->nasa_lo[7 * k + i]) || !std::isfinite(d->nasa_hi[7 * k + i])) {
        set_error("species %d has non-finite NASA coefficients", k);
        return CHEM_EINVAL;
      }
  }
  for (int j = 0; j < nr; ++j) {
    if (d->rtype[j] < 0 || d->rtype[j] > 2) { set_error("reaction %d: bad type", j); return CHEM_EINVAL; }
    int nre = 0, npr = 0;
    for (int i = 0; i < 3; ++i) {
      int a = d->reac[3 * j + i], b = d->prod[3 * j + i];
      if (a < -1 || a >= ns || b < -1 || b >= ns) {
        set_error("reaction %d: species index out of range", j);
        return CHEM_EINVAL;
      }
      nre += a >= 0; npr += b >= 0;
    }
    if (nre == 0 || npr == 0) { set_error("reaction %d: empty side", j); return CHEM_EINVAL; }
    if (!(d->A[j] >= 0.0) || !std::isfinite(d->b[j]) || !std::isfinite(d->Ea[j])) {
      set_error("reaction %d: bad Arrhenius parameters", j);
      return CHEM_EINVAL;
    }
    if (d->rtype[j] != 0)
      for (int k = 0; k < ns; ++k) {
        const double e = d->eff[(size_t)j * ns + k];
        if (!(e >= 0.0) || !std::isfinite(e)) {
          set_error("reaction %d: third-body efficiency of species %d is negative or not finite", j, k);
          return CHEM_EINVAL;
        }
      }
    if (d->rtype[j] == 2) {
      const double* t = d->troe + 7 * j;
      bool finite = true;
      for (int i = 0; i < 7; ++i) finite = finite && std::isfinite(t[i]);
      if (!finite || !(t[0] >= 0.0) || !(t[4] > 0.0) || !(t[5] > 0.0) ||
          (d->has_t2[j] != 0 && d->has_t2[j] != 1)) {
        set_error("reaction %d: bad Troe parameters", j);
        return CHEM_EINVAL;
      }
    }
  }
  return CHEM_OK;
}

}  // namespace

PoolUse::PoolUse() {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) { cudaGetLastError(); return; }
  Pools& P = pools();
  std::lock_guard<std::mutex> lk(P.mu);
  if (PoolSlot* s = pool_slot(P, dev)) {
    device = dev;
    context = s->context;
    ++s->users;
  }
}
PoolUse::~PoolUse() {
  if (device < 0) return;
  Pools& P = pools();
  std::lock_guard<std::mutex> lk(P.mu);
  for (PoolSlot& s : P.slot) {
    if (s.device != device || s.context != context) continue;
    if (--s.users > 0) return;
    int here = 0;
    if (cudaGetDevice(&here) != cudaSuccess) { cudaGetLastError(); return; }
    if (here != device && cudaSetDevice(device) != cudaSuccess) { cudaGetLastError(); return; }
    if (s.pool && context_number(device) == context) cudaMemPoolTrimTo(s.pool, 0);
    if (here != device) cudaSetDevice(here);
    return;
  }
}

cudaError_t ws_alloc(void** p, size_t bytes, cudaStream_t stream) {
  cudaMemPool_t pool = device_pool();
  if (pool) {
    const cudaError_t e = cudaMallocFromPoolAsync(p, bytes, pool, stream);
    if (e == cudaSuccess || e == cudaErrorMemoryAllocation) return e;
    cudaGetLastError();                // the default pool serves
  }
  return cudaMallocAsync(p, bytes, stream);
}
}  // namespace chem

using namespace chem;

extern "C" int chem_load_mechanism_desc(const chem_mech_desc* desc, chem_mech_t* out) {
  if (!out) { set_error("NULL output handle"); return CHEM_EINVAL; }
  *out = nullptr;
  int rc = validate(desc);
  if (rc) return rc;
  chem_mech_s* m = new (std::nothrow) chem_mech_s();
  if (!m) { set_error("out of host memory"); return CHEM_ENOMEM; }
  rc = build(desc, m);
  if (rc) { chem_free_mechanism(m); return rc; }
  *out = m;
  return CHEM_OK;
}

extern "C" int chem_load_mechanism(const char* path, chem_mech_t* out) {
  if (!path || !out) { set_error("NULL argument"); return CHEM_EINVAL; }
  std::ifstream f(path);
  if (!f) { set_error("cannot open %s", path); return CHEM_ENOTFOUND; }
  std::stringstream ss;
  ss << f.rdbuf();
  std::istringstream in(ss.str());
  std::string tok;
  auto expect = [&](const char* w) { return (in >> tok) && tok == w; };
  int ne = 0, ns = 0, nr = 0, ver = 0;
  std::string name;
  if (!expect("CHEMMECH") || !(in >> ver) || ver != 1 || !expect("name") || !(in >> name) ||
      !expect("elements") || !(in >> ne) || ne < 1 || ne > 64) {
    set_error("%s: bad CHEMMECH header", path);
    return CHEM_EINVAL;
  }
  std::vector<double> emass(ne);
  for (int e = 0; e < ne; ++e)
    if (!(in >> tok >> emass[e])) { set_error("%s: bad element line", path); return CHEM_EINVAL; }
  if (!expect("species") || !(in >> ns) || ns < 1 || ns > 4096) {
    set_error("%s: bad species header", path);
    return CHEM_EINVAL;
  }
  std::vector<int> comp((size_t)ns * ne);
  std::vector<double> lo(7 * ns), hi(7 * ns);
  for (int k = 0; k < ns; ++k) {
    in >> tok;
    for (int e = 0; e < ne; ++e) in >> comp[(size_t)k * ne + e];
    for (int i = 0; i < 7; ++i) in >> lo[7 * k + i];
    for (int i = 0; i < 7; ++i) in >> hi[7 * k + i];
    if (!in) { set_error("%s: bad species %d", path, k); return CHEM_EINVAL; }
  }
  if (!expect("reactions") || !(in >> nr) || nr < 0 || nr > 30000) {
    set_error("%s: bad reactions header", path);
    return CHEM_EINVAL;
  }
  std::vector<int> rtype(nr), reac(3 * nr), prod(3 * nr), has_t2(nr, 0);
  std::vector<double> A(nr), b(nr), Ea(nr), troe(7 * (size_t)nr, 0.0), eff((size_t)nr * ns, 1.0);
  for (int j = 0; j < nr; ++j) {
    in >> rtype[j];
    for (int i = 0; i < 3; ++i) in >> reac[3 * j + i];
    for (int i = 0; i < 3; ++i) in >> prod[3 * j + i];
    in >> A[j] >> b[j] >> Ea[j];
    if (rtype[j] == 2) {
      for (int i = 0; i < 7; ++i) in >> troe[7 * j + i];
      in >> has_t2[j];
    }
    if (rtype[j] != 0) {
      int n = 0;
      in >> n;
      for (int i = 0; i < n && in; ++i) {
        int k = -1;
        double v = 0;
        in >> k >> v;
        if (k < 0 || k >= ns) { set_error("%s: reaction %d efficiency index", path, j); return CHEM_EINVAL; }
        eff[(size_t)j * ns + k] = v;
      }
    }
    if (!in) { set_error("%s: bad reaction %d", path, j); return CHEM_EINVAL; }
  }
  if (!expect("end")) { set_error("%s: missing end", path); return CHEM_EINVAL; }
  chem_mech_desc d{};
  d.n_species = ns; d.n_elements = ne; d.n_reactions = nr;
  d.elem_mass = emass.data(); d.comp = comp.data(); d.nasa_lo = lo.data(); d.nasa_hi = hi.data();
  d.rtype = rtype.data(); d.reac = reac.data(); d.prod = prod.data(); d.A = A.data();
  d.b = b.data(); d.Ea = Ea.data(); d.troe = troe.data(); d.has_t2 = has_t2.data();
  d.eff = eff.data();
  return chem_load_mechanism_desc(&d, out);
}

extern "C" int chem_free_mechanism(chem_mech_t m) {
  if (!m) { set_error("NULL mechanism"); return CHEM_EINVAL; }
  if (m->d_blob) cudaFree(m->d_blob);
  if (m->d_jac) cudaFree(m->d_jac);
  if (m->d_fx) cudaFree(m->d_fx);
  if (m->d_co) cudaFree(m->d_co);
  if (m->d_tab) cudaFree(m->d_tab);
  if (m->d_gx) cudaFree(m->d_gx);
  if (m->d_gxj) cudaFree(m->d_gxj);
  delete m;
  return CHEM_OK;
}

extern "C" int chem_mechanism_info(chem_mech_t m, int* n_species, int* n_reactions,
                                   int* n_elements) {
  if (!m) { set_error("NULL mechanism"); return CHEM_EINVAL; }
  if (n_species) *n_species = m->ns;
  if (n_reactions) *n_reactions = m->nr;
  if (n_elements) *n_elements = m->ne;
  return CHEM_OK;
}

extern "C" const char* chem_last_error(void) { return chem::g_err.c_str(); }
