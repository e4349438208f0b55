// coupled_prox.cuh -- the joint proximal half-steps of the steps with several
// couplings (Sec. 5.2, 5.3) at one cell, as the CUDA-core forms (attraction.cu,
// strip.cu) apply them.
#pragma once

#include "jko_internal.cuh"

namespace jko {

// Wasserstein attraction: p = Prox_{sigma' h} at the geometric mean
// s_1^{w1} s_2^{w2} (w1 = 1/(1+tau), w2 = tau/(1+tau)), a_m = p / s_m.  0 where
// either s vanishes.
template <typename T, int EK>
__device__ __forceinline__ void attraction_cell(const ProxArgs<T>& P, int idx, T x1, T x2, T w1,
                                                T w2, T& a1, T& a2, T& p) {
  const T g = (x1 > T(0) && x2 > T(0))
                  ? dev_exp<T>(w1 * dev_log<T>(x1) + w2 * dev_log<T>(x2)) : T(0);
  p = prox_ratio<T, EK>(P, idx, g) * g;
  // a_m = p / s_m with IEEE division: s_m may be subnormal far from the
  // support of b_m, where x * rcp(s) would overflow (a_m itself stays finite,
  // ~ (s_other / s_m)^{weight})
  a1 = x1 > T(0) ? p / x1 : T(0);
  a2 = x2 > T(0) ? p / x2 : T(0);
}

// Two densities coupled through the congestion of their sum (Sec. 5.3): with
// a~_m = s_m e^{-sigma w_m}, p_m = a~_m min(1, kappa / (a~_1 + a~_2)) and
// a_m = p_m / s_m = e^{-sigma w_m} min(1, ...) (no division by s_m).
template <typename T>
__device__ __forceinline__ void species_cell(T s1, T s2, T e1, T e2, T kappa, int has_kappa, T& a1,
                                             T& a2, T& p1, T& p2) {
  const T t1 = s1 * e1, t2 = s2 * e2;
  const T t = t1 + t2;
  const T f = (has_kappa && t > kappa) ? kappa / t : T(1);
  a1 = e1 * f;
  a2 = e2 * f;
  p1 = t1 * f;
  p2 = t2 * f;
}

// Weighted geometric mean x^{1/(1+t)} y^{t/(1+t)}, 0 where either vanishes.
template <typename T>
__device__ __forceinline__ T weighted_geomean(T x, T y, T t) {
  return (x > T(0) && y > T(0)) ? dev_exp<T>((dev_log<T>(x) + t * dev_log<T>(y)) / (T(1) + t))
                                : T(0);
}

// p / s with IEEE division, 0 where p = 0 (s may be subnormal in the far field)
template <typename T>
__device__ __forceinline__ T safe_ratio(T p, T s) {
  return (p > T(0) && s > T(0)) ? p / s : T(0);
}

// min(e g(x, y), kappa): the common marginal of two couplings of the pairwise attraction.
template <typename T>
__device__ __forceinline__ T pairwise_marginal(T x, T y, T t, T e, T kappa, int has_kappa) {
  T pm = weighted_geomean<T>(x, y, t) * e;
  if (has_kappa && pm > kappa) pm = kappa;
  return pm;
}

}  // namespace jko
