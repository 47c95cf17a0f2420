// The integrator with one thread per cell (small mechanisms; what bounds it and why: see
// integrator_cell.cuh).  A warp runs its 32 cells in lockstep, one Rodas4 attempt per pass; a lane
// whose cell is done claims the next one from the work queue at the next pass (one atomicAdd per
// warp for all lanes that need a cell), so cells of different sub-step counts do not wait for each
// other.
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <algorithm>

#include "chem_internal.h"
#include "integrator_cell.cuh"

namespace chem {

// several lanes per cell (integrator_coop.cu)
int cell_lanes(const chem_mech_s* m, int64_t ncells, int ctas, int smem_max);
int launch_coop_advance(const chem_mech_s* m, const QueueParams& Q, int lanes, int sms, int smem_max, int max_ctas,
                        cudaStream_t stream);

namespace {

using cell::Ws;

struct CellParams {
  FxLayout fx;
  MechLayout lay;
  const unsigned char *fxblob, *blob;
  QueueParams q;
  double* mx;                  // WIDE: the matrices, a warp's N x N x 32 after the other's
};

struct CellEvalParams {
  FxLayout fx;
  MechLayout lay;
  const unsigned char *fxblob, *blob;
  const double *T, *p, *Y;
  int64_t ld, ncells;
  double *f, *J;
};

__device__ __forceinline__ void stage(const unsigned char* src, unsigned char* dst, int bytes) {
  const int4* s = (const int4*)src;
  int4* d = (int4*)dst;
  for (int i = threadIdx.x; i < bytes / 16; i += blockDim.x) d[i] = __ldg(s + i);
}

// One Rodas4 attempt of the lane's cell with step h: false on an exactly singular iteration
// matrix; otherwise e2 = the squared weighted RMS error and the new state left in U_5's place
// (elements U + 5 N ..: y_new), which the caller copies on acceptance.
template <int NS>
__device__ __forceinline__ bool attempt(const cell::View& m, double* col, double* M, double p, double invp, double h, double rtol,
                                        double atol, double* e2) {
  using w = Ws<NS>;
  constexpr int N = w::N;
  const double invh = fx::rcp(h), ig = invh * (1.0 / kGamma);
  cell::rhs<NS, true>(m, col, M, col[w::Y * 32], [&](int k) { return col[(w::Y + 1 + k) * 32]; }, p, invp, w::U);
#pragma unroll
  for (int i = 0; i < N; ++i) M[i * (N + 1) * 32] += ig;

  // LU with partial pivoting, rows in place: row[i] is the offset of logical row i (32-bit shared
  // offsets in registers).  Column k's candidates stay in registers, the pivot search runs on the
  // integer pipe, U's diagonal is stored as its reciprocal.
  int row[N];
#pragma unroll
  for (int i = 0; i < N; ++i) row[i] = i * N * 32;
  bool singular = false;
#pragma unroll
  for (int k = 0; k < N; ++k) {
    double v[N];
    unsigned long long best = 0ull;
    int bi = k;
#pragma unroll
    for (int i = k; i < N; ++i) {
      v[i] = M[row[i] + k * 32];
      const unsigned long long key = pivot_key(v[i]);
      if (key > best) { best = key; bi = i; }
    }
    if (best == 0ull) singular = true;
    double piv = v[k];
    int rp = row[k];
#pragma unroll
    for (int i = k + 1; i < N; ++i)
      if (i == bi) {
        piv = v[i]; v[i] = v[k];
        rp = row[i]; row[i] = row[k];
      }
    row[k] = rp;
    const double ip = fx::rcp(piv);
    M[rp + k * 32] = ip;
    double u[N];
#pragma unroll
    for (int j = k + 1; j < N; ++j) u[j] = M[rp + j * 32];
#pragma unroll
    for (int i = k + 1; i < N; ++i) {
      const double l = v[i] * ip;
      double* r = M + row[i];
      r[k * 32] = l;
#pragma unroll
      for (int j = k + 1; j < N; ++j) r[j * 32] = fma(-l, u[j], r[j * 32]);
    }
  }

#pragma unroll 1
  for (int s = 0; s < 6; ++s) {
    const int us = w::U + s * N;
    if (s > 0) {
      const double* ra = kRA[s];
      auto stage_value = [&](int i) {
        double v = col[(w::Y + i) * 32];
        for (int j = 0; j < s; ++j) v = fma(ra[j], col[(w::U + j * N + i) * 32], v);
        return v;
      };
      cell::rhs<NS, false>(m, col, M, stage_value(0), [&](int k) { return stage_value(1 + k); }, p, invp, us);
    }
    // right-hand side f + sum_j (C_sj / h) u_j, then both triangular sweeps in registers
    double b[N], t[N];
#pragma unroll
    for (int i = 0; i < N; ++i) b[i] = col[(us + i) * 32];
    for (int j = 0; j < s; ++j) {
      const double c = kRC[s][j] * invh;
#pragma unroll
      for (int i = 0; i < N; ++i) b[i] = fma(c, col[(w::U + j * N + i) * 32], b[i]);
    }
#pragma unroll
    for (int i = 0; i < N; ++i) col[(us + i) * 32] = b[i];
#pragma unroll
    for (int i = 0; i < N; ++i) {
      // row[i] = physical row * N * 32: the permuted right-hand side
      double v = col[us * 32 + row[i] / N];
#pragma unroll
      for (int k = 0; k < i; ++k) v = fma(-M[row[i] + k * 32], t[k], v);
      t[i] = v;
    }
#pragma unroll
    for (int i = N - 1; i >= 0; --i) {
      double v = t[i];
#pragma unroll
      for (int k = N - 1; k > i; --k) v = fma(-M[row[i] + k * 32], t[k], v);
      t[i] = v * M[row[i] + i * 32];
    }
#pragma unroll
    for (int i = 0; i < N; ++i) col[(us + i) * 32] = t[i];
  }
  double acc = 0.0;
#pragma unroll
  for (int i = 0; i < N; ++i) {
    const double y = col[(w::Y + i) * 32];
    double v = y;
#pragma unroll
    for (int s = 0; s < 6; ++s) v = fma(kRM[s], col[(w::U + s * N + i) * 32], v);
    const double sc = fma(rtol, fx::max_pos(fabs(y), fabs(v)), atol);
    const double r = col[(w::U + 5 * N + i) * 32] * fx::rcp(sc);
    acc = fma(r, r, acc);
    col[(w::U + 5 * N + i) * 32] = v;
  }
  *e2 = acc * (1.0 / N);
  return !singular;
}

// WIDE: eight warps an SM instead of four.  Four hold their whole workspace in shared memory (51 KB a
// warp for 9 species) and keep the FP64 pipe 64 % busy: a sub-partition's one warp cannot overlap its
// integer work with its own FP64 instructions.  With the matrix (half of the workspace) in an
// L2-resident array of global memory (25 KB a warp, 31 MB in all) two warps share a sub-partition:
// 2^20 flame cells 108 -> 80.2 ms.  (The vectors in global memory and the matrix in shared memory: 92.9.)
template <int NS, bool WIDE>
__global__ void __launch_bounds__(WIDE ? 256 : 128, 1) cell_advance_kernel(const __grid_constant__ CellParams P) {
  using w = Ws<NS>;
  constexpr int N = w::N;
  extern __shared__ __align__(16) unsigned char smem[];
  if (P.q.ncells_dev && *P.q.ncells_dev == 0u) return;     // an empty fallback pass
  stage(P.fxblob, smem, P.fx.bytes);
  __syncthreads();
  const cell::View m = cell::bind(smem, P.fx, P.blob, &P.lay);
  const int lane = threadIdx.x & 31;
  const int wib = threadIdx.x >> 5;
  double* const sh = (double*)(smem + P.fx.bytes);
  double* const col = sh + (size_t)wib * (WIDE ? w::VEC : w::TOTAL) * 32 + lane;
  double* const Mx = WIDE ? P.mx + ((size_t)blockIdx.x * (blockDim.x >> 5) + wib) * N * N * 32 + lane
                          : col + w::VEC * 32;
  auto dummy = [&] {
#pragma unroll
    for (int i = 0; i < N; ++i) col[(w::Y + i) * 32] = i == 0 ? 1000.0 : 1.0 / NS;
  };
  dummy();
  const long long total = P.q.ncells_dev ? min((long long)*P.q.ncells_dev, (long long)P.q.segs[0].ncells)
                                         : P.q.total_chunks;
  const unsigned long long t0 = P.q.budget_ns > 0 ? global_ns() : 0ull;
  const Segment* S = &P.q.segs[0];
  int64_t at = 0;
  bool active = false, exhausted = false;
  double dt = 1.0, rtol = 1e-6, atol = 1e-10, p = 1.0e6, invp = 1.0e-6, t = 0.0, h = 1.0, facmax = 6.0;
  int attempts = 0, nacc = 0, nrej = 0;

  for (;;) {
    // ---- lanes without a cell claim the next ones of the queue (warp-wide) ----
    for (;;) {
      const unsigned need = __ballot_sync(0xffffffffu, !active && !exhausted);
      if (need == 0u) break;
      const int leader = __ffs(need) - 1;
      unsigned long long base = 0ull;
      if (lane == leader) {
        // a time-sliced launch stops claiming once its budget is spent or its caller asks it to
        // stop: the cells claimed so far are exactly the prefix [0, counter) of the queue
        bool stop = false;
        if (P.q.budget_ns > 0) {
          const unsigned long long el = global_ns() - t0;
          stop = el > P.q.budget_ns ||
                 (P.q.stop && el > P.q.min_ns && *(const volatile unsigned int*)P.q.stop != 0u);
        }
        base = stop ? ~0ull : atomicAdd(P.q.counter, (unsigned long long)__popc(need));
      }
      base = __shfl_sync(0xffffffffu, base, leader);
      if (!active && !exhausted) {
        const unsigned long long mine = base + (unsigned long long)__popc(need & ((1u << lane) - 1u));
        if (base == ~0ull || mine >= (unsigned long long)total) {
          exhausted = true;
        } else {
          S = segment_of(P.q, (long long)mine);
          at = cell_of(S, (long long)mine - S->chunk_begin, 0);
          p = S->p[at];
          bool bad = !isfinite(p) || !(p > 0.0);
          double y[N];
          y[0] = S->T[at];
#pragma unroll
          for (int k = 0; k < NS; ++k) y[1 + k] = S->Y[(int64_t)k * S->ld + at];
          bad = bad || !(y[0] > 0.0);
#pragma unroll
          for (int i = 0; i < N; ++i) bad = bad || !isfinite(y[i]);
          if (bad) {                                  // the cell is left unchanged
            if (S->status) S->status[at] = (int8_t)CHEM_CELL_NONFINITE;
            if (S->nsub) S->nsub[at] = 0;
            if (S->nrej) S->nrej[at] = 0;
            p = 1.0e6;
          } else {
#pragma unroll
            for (int i = 0; i < N; ++i) col[(w::Y + i) * 32] = y[i];
            active = true;
            invp = 1.0 / p;
            dt = S->dt; rtol = S->rtol; atol = S->atol;
            t = 0.0; h = dt; facmax = 6.0;
            attempts = 0; nacc = 0; nrej = 0;
          }
        }
      }
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
    const bool ok = attempt<NS>(m, col, Mx, p, invp, run ? h : dt, rtol, atol, &e2);
    if (run) {
      if (!ok) {
        stop = true; status = CHEM_CELL_SINGULAR_LU;
      } else {
        ++attempts;
        const double fac = fx::step_factor(e2, m.e2, m.rc, m.lg);
        if (e2 <= 1.0) {
#pragma unroll
          for (int i = 0; i < N; ++i) col[(w::Y + i) * 32] = col[(w::U + 5 * N + i) * 32];
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
      S->T[at] = col[w::Y * 32];
#pragma unroll
      for (int k = 0; k < NS; ++k) S->Y[(int64_t)k * S->ld + at] = col[(w::Y + 1 + k) * 32];
      if (S->status) S->status[at] = (int8_t)status;
      if (S->nsub) S->nsub[at] = nacc;
      if (S->nrej) S->nrej[at] = nrej;
      active = false;
      dummy();
    }
    __syncwarp();
  }
}

// the right-hand side and Jacobian of chem_eval_rhs_jac with the integrator's device code
template <int NS>
__global__ void __launch_bounds__(128, 1) cell_eval_kernel(const __grid_constant__ CellEvalParams P) {
  using w = Ws<NS>;
  constexpr int N = w::N;
  extern __shared__ __align__(16) unsigned char smem[];
  stage(P.fxblob, smem, P.fx.bytes);
  __syncthreads();
  const cell::View m = cell::bind(smem, P.fx, P.blob, &P.lay);
  double* col = (double*)(smem + P.fx.bytes) + (size_t)(threadIdx.x >> 5) * w::TOTAL * 32 + (threadIdx.x & 31);
  for (int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; c < P.ncells; c += (int64_t)gridDim.x * blockDim.x) {
#pragma unroll
    for (int i = 0; i < N; ++i) col[(w::Y + i) * 32] = i == 0 ? P.T[c] : P.Y[(int64_t)(i - 1) * P.ld + c];
    const double p = P.p[c];
    auto Yk = [&](int k) { return col[(w::Y + 1 + k) * 32]; };
    if (P.J) cell::rhs<NS, true>(m, col, col + w::VEC * 32, col[w::Y * 32], Yk, p, 1.0 / p, w::U);
    else cell::rhs<NS, false>(m, col, col + w::VEC * 32, col[w::Y * 32], Yk, p, 1.0 / p, w::U);
    for (int i = 0; i < N; ++i) P.f[(int64_t)i * P.ld + c] = col[(w::U + i) * 32];
    if (P.J)
      for (int e = 0; e < N * N; ++e) P.J[(int64_t)e * P.ld + c] = -col[(w::VEC + e) * 32];
  }
}

struct Shape {
  int warps, sms;
  int smem_max;         // of a block, and the kernels' attribute whatever a launch takes: it is state of the
                        // function, and another thread may launch one of another size meanwhile
  size_t smem;          // of `warps` warps
};

// Warps of 32 cells whose whole workspace fits in an SM's shared memory, at most four: one per
// sub-partition (an FP64 instruction's latency equals its occupancy of the pipe), a fifth shares one.
// Three warps still issue at 89 % of four's FP64 rate (21.4 SM cycles an instruction against 19.0);
// two would leave half of the sub-partitions idle, so such mechanisms keep the group kernels.
template <int NS>
int shape_of(const chem_mech_s* m, Shape* s) {
  int dev = 0, smem_max = 0;
  CHEM_CUDA_TRY(cudaGetDevice(&dev));
  CHEM_CUDA_TRY(cudaDeviceGetAttribute(&smem_max, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
  CHEM_CUDA_TRY(cudaDeviceGetAttribute(&s->sms, cudaDevAttrMultiProcessorCount, dev));
  const size_t per = (size_t)Ws<NS>::TOTAL * 256;
  s->smem_max = smem_max;
  const long long room = (long long)smem_max - m->fx.bytes;
  s->warps = (int)std::min<long long>(4, room / (long long)per);
  s->smem = (size_t)m->fx.bytes + per * std::max(s->warps, 0);
  return CHEM_OK;
}

template <int NS>
int advance_t(const chem_mech_s* m, const QueueParams& Q, bool scratch, const chem_options* opt, cudaStream_t stream) {
  Shape s;
  int rc = shape_of<NS>(m, &s);
  if (rc) return rc;
  if (s.warps < 1) { set_error("mechanism too large for shared memory"); return CHEM_EINVAL; }
  CHEM_CUDA_TRY(cudaFuncSetAttribute((cell_advance_kernel<NS, false>), cudaFuncAttributeMaxDynamicSharedMemorySize, s.smem_max));
  const size_t per = (size_t)Ws<NS>::TOTAL * 256;
  int warps = s.warps;
  if (opt && opt->groups_per_cta > 0) warps = std::min(warps, (opt->groups_per_cta + 31) / 32);
  // fewer warps of cells than the GPU holds: spread them over the SMs
  const int64_t need = std::max<int64_t>(1, (Q.total_chunks + 31) / 32);
  warps = (int)std::min<int64_t>(warps, (need + s.sms - 1) / s.sms);
  int64_t grid = std::min<int64_t>(s.sms, (need + warps - 1) / warps);
  if (opt && opt->max_ctas > 0) grid = std::min<int64_t>(grid, opt->max_ctas);
  CellParams P;
  P.fx = m->fx; P.lay = m->lay; P.fxblob = (const unsigned char*)m->d_fx; P.blob = (const unsigned char*)m->d_blob;
  P.q = Q;
  // eight warps an SM (seven for 10 and 11 species) from 13 warps of cells an SM on (63 k cells on 152 SMs): below, the stiffest cells
  // of the last warps count for more than the rate (H2 flame, four / eight warps: 40009 cells 9.7 /
  // 12.6 ms, 80021 16.7 / 14.4, 2^20 108 / 80.2).  Without room for the matrices: four.
  constexpr size_t kMat = (size_t)Ws<NS>::N * Ws<NS>::N * 256, kVec = (size_t)Ws<NS>::VEC * 256;
  const int ww = (int)std::min<long long>(8, ((long long)s.smem_max - m->fx.bytes) / (long long)kVec);
  P.mx = nullptr;
  if (scratch && warps == s.warps && ww > warps && need >= 13 * grid) {
    const size_t wide = (size_t)m->fx.bytes + kVec * (size_t)ww;
    if (ws_alloc((void**)&P.mx, kMat * (size_t)ww * (size_t)grid, stream) == cudaSuccess) {
      cudaError_t e = cudaFuncSetAttribute((cell_advance_kernel<NS, true>), cudaFuncAttributeMaxDynamicSharedMemorySize,
                                           s.smem_max);
      if (e == cudaSuccess) {
        cell_advance_kernel<NS, true><<<(unsigned)grid, 32 * ww, wide, stream>>>(P);
        e = cudaGetLastError();
      }
      const cudaError_t fe = cudaFreeAsync(P.mx, stream);
      CHEM_CUDA_TRY(e);
      CHEM_CUDA_TRY(fe);
      return CHEM_OK;
    }
    (void)cudaGetLastError();
  }
  cell_advance_kernel<NS, false><<<(unsigned)grid, 32 * warps, (size_t)m->fx.bytes + per * warps, stream>>>(P);
  CHEM_CUDA_TRY(cudaGetLastError());
  return CHEM_OK;
}

template <int NS>
int eval_t(const chem_mech_s* m, const double* T, const double* p, const double* Y, int64_t ld, int64_t n, double* f,
           double* J, cudaStream_t stream) {
  Shape s;
  int rc = shape_of<NS>(m, &s);
  if (rc) return rc;
  CHEM_CUDA_TRY(cudaFuncSetAttribute(cell_eval_kernel<NS>, cudaFuncAttributeMaxDynamicSharedMemorySize, s.smem_max));
  CellEvalParams P;
  P.fx = m->fx; P.lay = m->lay; P.fxblob = (const unsigned char*)m->d_fx; P.blob = (const unsigned char*)m->d_blob;
  P.T = T; P.p = p; P.Y = Y; P.ld = ld; P.ncells = n; P.f = f; P.J = J;
  const int64_t grid = std::min<int64_t>((n + 32 * s.warps - 1) / (32 * s.warps), 65535);
  cell_eval_kernel<NS><<<(unsigned)grid, 32 * s.warps, s.smem, stream>>>(P);
  CHEM_CUDA_TRY(cudaGetLastError());
  return CHEM_OK;
}

}  // namespace

// Whether the mechanism's cells run one per thread: it has a fixed-point form (its species count is one
// of the instances'), and at least three warps of cells fit on an SM (see shape_of).
bool cell_kernel_fits(const chem_mech_s* m) {
  static_assert(kCellMinNs == 8 && kCellMaxNs == 11, "the instances below, advance_t's and eval_t's");
  if (!m->fx.bytes) return false;
  Shape s{0, 0, 0, 0};
  int rc = CHEM_EINVAL;
  switch (m->ns) {
    case 8: rc = shape_of<8>(m, &s); break;
    case 9: rc = shape_of<9>(m, &s); break;
    case 10: rc = shape_of<10>(m, &s); break;
    case 11: rc = shape_of<11>(m, &s); break;
    default: return false;
  }
  return rc == CHEM_OK && s.warps >= 3;
}

// scratch: whether the launch may take device memory from the pool
int launch_cell_advance(const chem_mech_s* m, const QueueParams& Q, bool scratch, const chem_options* opt,
                        cudaStream_t stream) {
  int dev = 0, sms = 0, smem_max = 0;
  CHEM_CUDA_TRY(cudaGetDevice(&dev));
  CHEM_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  CHEM_CUDA_TRY(cudaDeviceGetAttribute(&smem_max, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
  const int max_ctas = opt ? opt->max_ctas : 0;
  const bool shaped = opt && opt->groups_per_cta > 0;
  const int lanes = shaped ? 1 : cell_lanes(m, Q.total_chunks, max_ctas > 0 ? std::min(sms, max_ctas) : sms, smem_max);
  if (lanes > 1) return launch_coop_advance(m, Q, lanes, sms, smem_max, max_ctas, stream);
  switch (m->ns) {
    case 8: return advance_t<8>(m, Q, scratch, opt, stream);
    case 9: return advance_t<9>(m, Q, scratch, opt, stream);
    case 10: return advance_t<10>(m, Q, scratch, opt, stream);
    case 11: return advance_t<11>(m, Q, scratch, opt, stream);
    default: set_error("no cell kernel for %d species", m->ns); return CHEM_EINVAL;
  }
}

int launch_cell_eval(const chem_mech_s* m, const double* T, const double* p, const double* Y, int64_t ld, int64_t n,
                     double* f, double* J, cudaStream_t stream) {
  switch (m->ns) {
    case 8: return eval_t<8>(m, T, p, Y, ld, n, f, J, stream);
    case 9: return eval_t<9>(m, T, p, Y, ld, n, f, J, stream);
    case 10: return eval_t<10>(m, T, p, Y, ld, n, f, J, stream);
    case 11: return eval_t<11>(m, T, p, Y, ld, n, f, J, stream);
    default: set_error("no cell kernel for %d species", m->ns); return CHEM_EINVAL;
  }
}

}  // namespace chem
