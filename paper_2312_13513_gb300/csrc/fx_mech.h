// Fixed-point form of a mechanism (formats: fixed.cuh), as the cell-per-thread integrator stages
// it into shared memory.  Built once per mechanism on the host; a mechanism with a number outside
// the formats' range has none (FxLayout::bytes = 0) and runs on the FP64 kernels, a single
// reaction outside it carries FxReac::slow and takes the FP64 rate expressions.
#pragma once
#include <stdint.h>

namespace chem {

// one reaction; species slots beyond nre / npr are 0 and unread
struct alignas(16) FxReac {
  int64_t lnA, beta, Ta;      // log2 A (Q11.52), b (Q7.56), Ea / (Rc ln 2) / 128 (Q11.52)
  double b, TaK;              // b and Ea / Rc in FP64, for the temperature derivative
  uint8_t re[3], pr[3];       // species of each side
  uint8_t nre, npr;
  uint8_t sp[6];              // net production: nnet distinct species ...
  int8_t nu[6];               // ... with their coefficients
  uint8_t nnet, type, slow;
  int8_t dnu;
  int16_t tb, troe;           // third-body set and Troe record, -1: none
};

struct alignas(16) FxTroe {
  int64_t lnA0, b0, Ta0;      // low-pressure limit, as FxReac
  double b0d, Ta0K;
  double a, iT3, iT1, T2, has_t2;
};

// one species in one temperature range; the polynomial variable is tau = T / 2^r (r = 10 below
// TMID, 12 above), all Q11.52 except gl (Q7.56)
struct FxSpecies {
  int64_t g[5], ga6, gl;      // g/RT/ln 2 = g(tau) + ga6 (128 / T) + gl log2 T
  int64_t h[5], ha6;          // h/RT
  int64_t c[5];               // cp/R
};

struct FxLayout {
  int ns, nr, ntb, bytes;     // bytes = 0: no fixed-point form
  int o_exp2, o_lg, o_rcp;    // tables of fixed.cuh
  int o_sp;                   // FxSpecies [2][ns]
  int o_W, o_invW;            // [ns]
  int o_nu;                   // double [16]: coefficient of code c is c - 8
  int o_reac, o_troe;
  int o_effv, o_eff;          // sparse (efficiency - 1); dense efficiencies [ntb][ns]
  int o_effidx, o_effoff;
  int64_t lpr0;               // log2(p_atm / R), Q11.52
};

constexpr int kFxR0 = 10, kFxR1 = 12;

}  // namespace chem
