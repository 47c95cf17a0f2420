// The integrator's work queue: what a launch advances, as the group kernels (integrator.cu) and
// the cell-per-thread kernel (integrator_cell.cu) share it.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "chem_internal.h"

namespace chem {

// One independent set of cells advanced by a launch: its own state arrays, step and
// tolerances, optional index list and outputs.  A launch walks the chunks of all its segments
// through one work queue (iteration-level batching of several requests).
struct Segment {
  double* T;
  const double* p;
  double* Y;
  int64_t ld, ncells;
  const int32_t* idx;
  int8_t* status;
  int32_t* nsub;
  int32_t* nrej;
  double dt, rtol, atol;
  long long chunk_begin;           // first queue entry of this segment
};

constexpr int kMaxSegs = kMaxSegsPerLaunch;   // segments per launch (kernel-parameter space)

struct QueueParams {
  Segment segs[kMaxSegs];
  int nseg;
  long long total_chunks;
  int max_steps;
  unsigned long long* counter;
  const unsigned int* ncells_dev;  // single segment: cell count read from device memory
  unsigned long long budget_ns = 0;  // > 0: stop claiming chunks this long after the group started
  // time-sliced launches: a nonzero *stop (device memory, set by the caller while the slice runs)
  // also stops the claiming, once the group has run min_ns
  const unsigned int* stop = nullptr;
  unsigned long long min_ns = 0;
};

__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

__device__ __forceinline__ int64_t cell_of(const Segment* S, long long base, int c) {
  return S->idx ? (int64_t)S->idx[base + c] : (int64_t)(base + c);
}

__device__ __forceinline__ const Segment* segment_of(const QueueParams& P, long long chunk) {
  int s = 0;
  while (s + 1 < P.nseg && P.segs[s + 1].chunk_begin <= chunk) ++s;
  return &P.segs[s];
}

// Rodas4 coefficients, transformed (u-variable) form:
//   (I/(gamma h) - J) u_s = f(y + sum_j A[s][j] u_j) + sum_j (C[s][j]/h) u_j,
//   y_new = y + sum_s M[s] u_s,  error = u_5.
static __constant__ double kRA[6][6] = {
    {0, 0, 0, 0, 0, 0},
    {1.544, 0, 0, 0, 0, 0},
    {0.9466785280815826, 0.2557011698983284, 0, 0, 0, 0},
    {3.314825187068521, 2.896124015972201, 0.9986419139977817, 0, 0, 0},
    {1.221224509226641, 6.019134481288629, 12.53708332932087, -0.6878860361058950, 0, 0},
    {1.221224509226641, 6.019134481288629, 12.53708332932087, -0.6878860361058950, 1.0, 0}};
static __constant__ double kRC[6][6] = {
    {0, 0, 0, 0, 0, 0},
    {-5.6688, 0, 0, 0, 0, 0},
    {-2.430093356833875, -0.2063599157091915, 0, 0, 0, 0},
    {-0.1073529058151375, -9.594562251023355, -20.47028614809616, 0, 0, 0},
    {7.496443313967647, -10.24680431464352, -33.99990352819905, 11.70890893206160, 0, 0},
    {8.083246795921522, -7.981132988064893, -31.52159432874371, 16.31930543123136,
     -6.058818238834054, 0}};
static __constant__ double kRM[6] = {1.221224509226641, 6.019134481288629, 12.53708332932087,
                                     -0.6878860361058950, 1.0, 1.0};
constexpr double kGamma = 0.25;

// Pivot key of a matrix entry: the bit pattern of |a| read as an unsigned integer.  For
// non-negative doubles the integer order is the numeric order, so the pivot search runs on the
// integer pipes instead of FP64 compares (the FP64 pipe is the scarce one).  NaN maps to 0.
__device__ __forceinline__ unsigned long long pivot_key(double a) {
  const unsigned long long k = (unsigned long long)__double_as_longlong(a) & 0x7fffffffffffffffull;
  return k > 0x7ff0000000000000ull ? 0ull : k;
}

}  // namespace chem
