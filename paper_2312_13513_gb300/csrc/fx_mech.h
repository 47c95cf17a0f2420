// Fixed-point form of a mechanism (formats: fixed.cuh), as the cell-per-thread integrator stages
// it into shared memory.  Built once per mechanism on the host; a mechanism with a number outside
// the formats' range has none (FxLayout::bytes = 0) and runs on the FP64 kernels, a single
// reaction outside it carries FxReac::slow and takes the FP64 rate expressions.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace chem {

// Signed constants that multiply a temperature quantity are stored biased (fx::biased).

// One reaction with at most two species per side.  Species are byte offsets k * 256 of a cell's
// workspace columns (32 lanes of 8 bytes); an empty slot is species ns, whose concentration reads
// 1 and whose Gibbs energy 0.  The net production goes to four distinct species: those of the
// reaction, padded with others at coefficient 0, so that the four updates never alias.
struct alignas(16) FxRate {
  int64_t lnA;                // log2 A (Q11.52); 2000: the FP64 rate expressions take the reaction
  uint64_t beta;              // b (Q7.56), biased
  uint64_t Ta;                // Ea / (Rc ln 2) / 128 (Q11.52), biased
  uint16_t c[4];              // two reactants, two products
  uint16_t w[4];              // species of the net production ...
  int16_t dnu, id, tb, troe;  // id: index in the FP64 form; third-body set and Troe record, -1: none
  double nu[4];               // ... and its coefficients
  double b, TaK;              // b and Ea / Rc, for the temperature derivative
};

// any reaction (up to three species per side, six net species): what FxRate cannot hold
struct alignas(16) FxReac {
  int64_t lnA;
  uint64_t beta, Ta;
  double b, TaK;
  uint8_t re[3], pr[3], nre, npr;   // species of each side
  uint8_t sp[6];                    // net production: nnet distinct species ...
  int8_t nu[6];                     // ... with their coefficients
  uint8_t nnet, type;
  int16_t dnu, id, tb, troe;
};

struct alignas(16) FxTroe {
  int64_t lnA0;               // low-pressure limit, as FxRate
  uint64_t b0, Ta0;
  double b0d, Ta0K;
  double a, iT3, iT1, T2, has_t2;
};

// one species in one temperature range; the polynomial variable is tau = T / 2^r (r = 10 below
// TMID, 12 above), all Q11.52 except gl (Q7.56); the leading coefficients g[4], h[4], c[4] and
// ga6, gl, ha6 are biased
struct FxSpecies {
  int64_t g[5], ga6, gl;      // g/RT/ln 2 = g(tau) + ga6 (128 / T) + gl log2 T
  int64_t h[5], ha6;          // h/RT
  int64_t c[5];               // cp/R
};

// Enthalpy h/(R W) (K mol/g) and heat capacity cp/(R W) of one species in one temperature range as
// polynomials in tau = T / 2^r, each scaled by the largest power of two at which the magnitudes of its
// terms sum to less than 2^62 (2^fh, 2^fc); the leading coefficients h[5] and c[4] are biased.
// cf: the heat capacity in FP32
struct FxEnthalpy {
  int64_t h[6], c[5];
  int32_t fh, fc;
  float cf[5], pad[3];
};

// Species counts with instances of the kernels of one thread and of several lanes per cell, and a blob of
// this form.  Beyond 11 fewer than three warps of cells fit in an SM's shared memory (integrator_cell.cu).
// Below 8 none is compiled: those mechanisms keep the two-lane groups, and the two were not compared there.
constexpr int kCellMinNs = 8, kCellMaxNs = 11;

struct FxLayout {
  int ns, ntb, bytes;         // bytes = 0: no fixed-point form
  int o_exp2, o_lg, o_rcp;    // tables of fixed.cuh
  int o_sp;                   // FxSpecies [2][ns]
  int o_W, o_invW;            // [ns]
  int o_nu;                   // double [16]: coefficient of code c is c - 8
  int o_rate, o_reac, o_troe;   // FxRate [n_plain + n_tb + n_fo] in that order, FxReac [n_gen]
  int n_plain, n_tb, n_fo, n_gen;
  int o_effv, o_eff;          // sparse (efficiency - 1); dense efficiencies [ntb][ns]
  int o_effidx, o_effoff;
  int64_t lpr0;               // log2(p_atm / R), Q11.52
};

// Gather form of a cell's sums for several lanes per cell (integrator_coop.cu), where one thread
// scatters: per species the terms of its production rate (reaction << 4 | (coefficient + 8)), per
// entry of d(wdot)/dC (negated) the terms coef * value, both in the order in which the one thread
// adds them.  Values: 4 j + slot the derivative of reaction j by its slot's species, 4 n + j - n_plain
// the collision partners' factor of reaction j.  Entries by falling term count.
struct CoTerm {
  double coef;
  int src, pad;
};
struct CoLayout {
  int bytes;                  // 0: none (a reaction outside FxRate)
  int n, nent, nval;          // FxRate records, entries, values
  int o_woff, o_wterm;        // int [ns + 1], [..]
  int o_eoff, o_epos, o_term; // int [nent + 1], row * N + column [nent], CoTerm [..]
};

// The same for the group kernels (integrator.cu): one lane per reaction, so the records are arrays;
// species slots are indices, ns in an empty one.
struct GxLayout {
  int ns, nr, ntb, npieces, bytes;      // bytes = 0: no fixed-point form
  int o_exp2, o_sp, o_W, o_invW, o_nu;
  int o_lnA, o_beta, o_Ta;              // [nr] as FxRate
  int o_reac, o_prod, o_rinfo;          // short4 [nr]: species; type, dnu, third-body set, Troe record
  int o_troe, o_effv, o_effidx, o_effoff;
  int o_wpk, o_pterm, o_poff;           // production lists, as MechLayout
  int64_t lpr0;
};

// Jacobian-assembly program of the group kernels with the fixed-point form (global memory).  The
// entries of d(wdot)/dC, sorted by their term counts, are dealt to the kGxLanes lanes of a group in
// chunks of kGxLanes; a chunk is as many term rows as its longest entry needs (terms of coefficient
// 0 fill the others), and term row r of lane t lies at r * kGxLanes + t, chunk after chunk: one
// coalesced stream that a lane can read ahead.  A lane's entry ends with the row whose z (slot) or
// y (part) is not -1: its place row << 16 | column.
// A slot term is the derivative of one direction of reaction j with respect to one of its species
// for one unit of net coefficient: x = (2 j + side) << 1 | (coefficient negative), a null term points
// at the zero behind the 2 nr derivatives; y = o1 | o2 << 16, the side's other species.
// Collision partners: d(wdot_k)/dC_m = sum_j nu_kj X_j eff_jm = R_k + sum_j nu_kj X_j (eff_jm - 1),
// with R_k = sum_j nu_kj X_j the same for every column: only the sparse deviations are terms
// (x = set, coefficient nu (eff - 1)); R_k (row_off, row_src = set << 4 | (nu + 8)) joins the chain
// rule.  For the 53-species mechanism this leaves 4.4 k slot and 2.8 k partner terms of 13.1 k.
constexpr int kGxLanes = 128;
constexpr int kGxUnroll = 4;                               // term rows are a multiple of this
struct GxJac {
  int nslot = 0, npart = 0;                                // term rows; of the first kind kGxUnroll at least
  const int4* slot = nullptr;
  const int2* part = nullptr;
  const double* part_coef = nullptr;
  const int *row_off = nullptr, *row_src = nullptr;        // [ns + 1], terms of R_k
};

constexpr int kFxR0 = 10, kFxR1 = 12;

}  // namespace chem
