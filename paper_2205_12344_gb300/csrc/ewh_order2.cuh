// Arithmetic of one order-2 level in 2D, every rounding written out: kernels that
// tile the grid differently give the same bits.
#pragma once

#include "ewh_internal.cuh"

namespace ewh {

__device__ __forceinline__ double o2_mul(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float o2_mul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double o2_fma(double a, double b, double c) { return __fma_rn(a, b, c); }
__device__ __forceinline__ float o2_fma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double o2_add(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ float o2_add(float a, float b) { return __fadd_rn(a, b); }

// Coefficients of the row of 2 h^2 rho M^{-1} K for one component: axis a along the
// component, b across; 0 / 1 the lower / upper neighbour.
template <typename T>
struct O2Row {
  T ca0, ca1, cb0, cb1;  // edges: twice the mean of lambda + 2 mu (along), mu (across)
  T la0, la1, mb0, mb1;  // mixed terms, half of lambda and mu at the neighbours
};

// Neighbour values: own component along and across, the other component at the corners.
template <typename T>
struct O2Vals {
  T a0, a1, b0, b1, v00, v01, v10, v11;  // v(a side)(b side)
};

template <typename T>
__device__ __forceinline__ T o2_row(const O2Row<T>& c, T u, const O2Vals<T>& n) {
  T k1 = o2_mul(c.ca0, o2_add(u, -n.a0)), k2 = o2_mul(c.la0, o2_add(n.v01, -n.v00));
  k1 = o2_fma(c.ca1, o2_add(u, -n.a1), k1);
  k2 = o2_fma(-c.la1, o2_add(n.v11, -n.v10), k2);
  k1 = o2_fma(c.cb0, o2_add(u, -n.b0), k1);
  k2 = o2_fma(c.mb0, o2_add(n.v10, -n.v00), k2);
  k1 = o2_fma(c.cb1, o2_add(u, -n.b1), k1);
  k2 = o2_fma(-c.mb1, o2_add(n.v11, -n.v01), k2);
  return o2_add(k1, k2);
}

// delta^{n+1} with k = o2_row, ks = kt / (2 rho h^2), kc = kt cos(w t_n); the first level
// (Taylor start) has half of ks and kc and d = 0.
template <typename T, bool FORCED>
__device__ __forceinline__ T o2_delta(T ks, T k, T kc, T fr, T d) {
  const T r = o2_fma(-ks, k, d);
  return FORCED ? o2_fma(-kc, fr, r) : r;
}

}  // namespace ewh
