// heat_cell.cuh -- the per-cell arithmetic of the heat kernel's Clenshaw recurrence
// (heat.cu, heat_tile.cu).
#pragma once

#include "jko_internal.cuh"

namespace jko {

// Block of the kernels per phase (small tiles: the work is FP64-bound per SM, so more blocks
// spread it), and the cells whose terms of the residual are added together first.
constexpr int HBX = 16, HBY = 8;

// ---- the per-cell arithmetic of the recurrence ----
// Written with explicit roundings, so that every kernel below (per phase or
// persistent) performs the same operations whatever the compiler contracts.
// The iterates W are FP64 for both precisions: a high-degree recurrence
// cancels large intermediate terms in the far field, where the kernel's tail
// is many orders below its peak, so single precision there costs digits (the
// flows' error grew 16-fold with FP32 iterates).  Double-float iterates (two
// floats, ~48 significant bits, on the FP32 pipe) were measured slower than
// FP64 on GB300 (100^2: 4.8k against 5.3k pairs/s): the stencil is bound by
// the latency of its dependent chains, which double-float arithmetic
// lengthens, not by the FP64 pipe's throughput.
template <typename T> struct HeatIter { using W = double; };

// constants and inputs as iterates
template <typename W> __device__ __forceinline__ W wc(double d) { return d; }
__device__ __forceinline__ double wv(double v) { return v; }
template <typename W> __device__ __forceinline__ W wzero() { return 0.0; }
// c v (the first iterate b_D = c_D v)
__device__ __forceinline__ double wscale(double c, double v) { return __dmul_rn(c, v); }

// One Clenshaw step's value ck v + 2 B b1 - b2, B = (A - theta Id) / delta.  With theta = 1 +
// delta and delta = 2 cx + 2 cy (the interval is [1, 1 + 4 cx + 4 cy]) the diagonal of B
// vanishes on an interior cell, and where a neighbour is missing (Neumann) the cell's own
// value takes its place: 2 B b1 = -ax (l + r) - ay (u + d), ax = 2 cx / delta, ay = 2 cy /
// delta (the closing step's B b1: half of both).  Five FP64 operations four deep, where the
// sum over differences c (b1_i - b1_j), less theta b1, scaled, took twelve nine deep.
__device__ __forceinline__ double cl_value(double ck, double v, double b2, double ax, double ay,
                                           double l, double r, double u, double d) {
  return __fma_rn(-ay, __dadd_rn(u, d), __fma_rn(-ax, __dadd_rn(l, r), __fma_rn(ck, v, -b2)));
}

// The operator's output is clamped at 0: xi~ is positive, and the expansion's
// error is normwise (~1e-15 of the largest entry), so where the true kernel
// tail lies below it the sum can come out slightly negative; 0 there is the
// same underflow the Gaussian kernel meets far from its support (the b-update
// and the prox treat it so).  NaN passes through.
template <typename T> __device__ __forceinline__ T close_out(double r) {
  return (T)(r < 0.0 ? 0.0 : r);
}

}  // namespace jko
