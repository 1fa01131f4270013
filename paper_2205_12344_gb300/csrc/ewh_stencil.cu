// Fused leapfrog + trapezoid-filter step kernels.
//
// One launch advances every right-hand side by one time level of the
// time-corrected explicit scheme (Section 4.3, eq. elastic-time-explicit-
// corrected), written in increment form
//     delta^{n+1} = delta^n - kt (M^{-1} K u^n + (f / rho) cos(w t_n)),
//     u^{n+1}     = u^n + delta^{n+1},
//     acc        += w_{n+1} u^{n+1}                (trapezoid filter, eq. qoper)
// with the Taylor start folded into the first launch:
//     delta^1 = -(kt/2) (M^{-1} K u^0 + f / rho),  acc = w_0 u^0 + w_1 u^1.
// K = -L_h is the Hessian of the discrete elastic energy (Section 4.1):
//   order 2: compact form; pure terms on edges with edge coefficients equal
//            to the mean of the two end nodes, mixed terms at nodes with
//            centred differences (one-sided on a free boundary node), the
//            trapezoid factor 1/2 per free side;
//   order 4: pointwise energy density with all first derivatives from the
//            fourth-order diagonal-norm summation-by-parts operator D; then
//            M^{-1} K u = (1/(rho h^2)) sum_a [ -D_a sigma_{.a} + H_a^{-1} B_a sigma_{.a} ].
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstdlib>
#include <cstring>

#include "ewh_internal.cuh"
#include "ewh_order2.cuh"

namespace ewh {

// The SBP boundary closure (SBP_CLOSURE) in constant memory.
#define EWH_SBP_ROW(T, r)                                                                         \
  {                                                                                               \
    (T)SBP_CLOSURE[r][0], (T)SBP_CLOSURE[r][1], (T)SBP_CLOSURE[r][2], (T)SBP_CLOSURE[r][3],        \
        (T)SBP_CLOSURE[r][4], (T)SBP_CLOSURE[r][5]                                                \
  }
__constant__ double c_sbp_d[4][6] = {EWH_SBP_ROW(double, 0), EWH_SBP_ROW(double, 1), EWH_SBP_ROW(double, 2),
                                     EWH_SBP_ROW(double, 3)};
__constant__ float c_sbp_f[4][6] = {EWH_SBP_ROW(float, 0), EWH_SBP_ROW(float, 1), EWH_SBP_ROW(float, 2),
                                    EWH_SBP_ROW(float, 3)};
#undef EWH_SBP_ROW

template <typename T>
__device__ __forceinline__ T sbp_coef(int r, int j);
template <>
__device__ __forceinline__ double sbp_coef<double>(int r, int j) { return c_sbp_d[r][j]; }
template <>
__device__ __forceinline__ float sbp_coef<float>(int r, int j) { return c_sbp_f[r][j]; }

// SBP first derivative along one axis at position p of a line of N nodes;
// v points at the node, s is the element stride along the axis.
template <typename T>
__device__ __forceinline__ T sbp_d1(const T* v, long long s, int p, int N) {
  if (p < 4) {
    T acc = T(0);
#pragma unroll
    for (int j = 0; j < 6; ++j) acc += sbp_coef<T>(p, j) * v[(long long)(j - p) * s];
    return acc;
  }
  if (p > N - 5) {
    const int r = N - 1 - p;
    T acc = T(0);
#pragma unroll
    for (int j = 0; j < 6; ++j) acc -= sbp_coef<T>(r, j) * v[(long long)(r - j) * s];
    return acc;
  }
  return (v[-2 * s] - T(8) * v[-s] + T(8) * v[s] - v[2 * s]) * T(1.0 / 12.0);
}

// interior row of the SBP first derivative (unit spacing): (1, -8, 0, 8, -1) / 12
template <typename T>
__device__ __forceinline__ T c4(T m2, T m1, T p1, T p2) {
  return (m2 - T(8) * m1 + T(8) * p1 - p2) * T(1.0 / 12.0);
}

// Programmatic dependent launch: a step kernel may start while the previous
// one drains.  Before pdl_wait() a kernel reads only data the solve never
// writes (lambda, mu, 1/(rho h^2), f/rho); pdl_wait() returns once the previous
// kernel has completed and its writes are visible; pdl_trigger() lets the next
// kernel begin launching.  Both are no-ops for a normal launch.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// ---------------------------------------------------------------------------
// Order 2, 2D: 32 x TYV tile, one node per thread, halo 1 in shared memory.  The
// medium is staged before the wait for the previous level.  Warps off the free sides
// take the row without weights; next to one, a difference takes the node itself
// for the neighbour that is missing, over half the width, and the transposed
// difference weighs its two members (ga, gb).
//
// Small grids are latency: 62^2 4.0 -> 1.4 us per level in FP32, 7.0 -> 3.7 us in FP64
// (medium staged early, fewer FP64 instructions: some 55 a node for 122).  Larger ones
// are bound by the FP64 pipe, in FP32 by L2 and HBM: 1024^2 214 -> 124 us and
// 19.7 -> 10.2 us, 2000^2 786 -> 474 us and 77 -> 54 us.
// ---------------------------------------------------------------------------
template <typename T, int MODE, bool FORCED, int TYV>
__global__ void __launch_bounds__(32 * TYV) step2d_o2(Geom g, WaveFields<T> f, StepScalars s) {
  if (g.dim != 2) return;
  constexpr int TX = 32, TY = TYV, SX = TX + 2, SY = TY + 2, PL = SX * SY;
  __shared__ T su[2 * PL], sl[PL], sm[PL];
  const int rhs = blockIdx.z;
  const int x0 = g.off[0] + blockIdx.x * TX, y0 = g.off[1] + blockIdx.y * TY;
  const int tid = threadIdx.y * TX + threadIdx.x;
  constexpr int NL = (PL + TX * TY - 1) / (TX * TY);
  int q[NL];  // padded offsets of the tile positions this thread stages
#pragma unroll
  for (int k = 0; k < NL; ++k) {
    const int i = tid + k * TX * TY, ly = i / SX;
    q[k] = (int)pidx(g, 0, 0, x0 - 1 + (i - ly * SX), y0 - 1 + ly, 0);
    if (i < PL) sl[i] = f.lam[q[k]], sm[i] = f.mu[q[k]];
  }
  const int x = x0 + threadIdx.x, y = y0 + threadIdx.y;
  const bool live = x < g.off[0] + g.nu[0] && y < g.off[1] + g.nu[1];
  const long long pc = pidx(g, 0, 0, x, y, 0), p = (long long)rhs * 2 * g.field + pc;
  T irh = T(0), fr[2] = {T(0), T(0)}, dl[2], ap[2];
  if (live) {
    irh = f.irh2[pc];
    if (FORCED) fr[0] = f.frho[p], fr[1] = f.frho[p + g.field];
  }
  pdl_wait();
  pdl_trigger();
  const T* const U = f.u_cur + (long long)rhs * 2 * g.field;
#pragma unroll
  for (int k = 0; k < NL; ++k) {
    const int i = tid + k * TX * TY;
    if (i < PL) su[i] = U[q[k]], su[PL + i] = U[g.field + q[k]];
  }
#pragma unroll
  for (int c = 0; c < 2; ++c) {
    const bool rd = live && (MODE == STEP_MID || MODE == STEP_LAST);
    dl[c] = rd ? f.delta[p + c * g.field] : T(0);
    ap[c] = rd ? f.acc[p + c * g.field] : T(0);
  }
  __syncthreads();
  const bool lo[2] = {x == 0, y == 0}, hi[2] = {x == g.n[0] - 1, y == g.n[1] - 1};
  // of the warp: one lane on a free side takes all of them through the general form
  const bool side = __any_sync(0xffffffffu, live && (lo[0] || hi[0] || lo[1] || hi[1]));
  if (!live) return;
  const int o = (threadIdx.y + 1) * SX + threadIdx.x + 1;
  const T l0 = sl[o], m0 = sm[o], p0 = l0 + T(2) * m0;
  const double kt = MODE == STEP_FIRST ? 0.5 * s.kt : s.kt;
  const T ks = T(0.5 * kt) * irh, kc = FORCED ? T(kt * s.cosn) : T(0);
  auto node = [&](auto tag) {
    constexpr bool SIDE = decltype(tag)::value;
    int nb[2][2] = {{-1, 1}, {-SX, SX}};
    T w[2] = {T(1), T(1)}, ga[2], gb[2];
    if (SIDE) {
#pragma unroll
      for (int a = 0; a < 2; ++a) {
        w[a] = lo[a] || hi[a] ? T(2) : T(1);
        ga[a] = lo[a] ? T(-2) : w[a];
        gb[a] = hi[a] ? T(-2) : w[a];
        if (lo[a]) nb[a][0] = 0;
        if (hi[a]) nb[a][1] = 0;
      }
    }
    T lam[2][2], mu[2][2];
#pragma unroll
    for (int a = 0; a < 2; ++a)
#pragma unroll
      for (int e = 0; e < 2; ++e) lam[a][e] = sl[o + nb[a][e]], mu[a][e] = sm[o + nb[a][e]];
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      const int b = 1 - c;
      const T *const u = su + c * PL + o, *const v = su + b * PL + o;
      O2Row<T> r{p0 + (lam[c][0] + T(2) * mu[c][0]), p0 + (lam[c][1] + T(2) * mu[c][1]), m0 + mu[b][0], m0 + mu[b][1],
                 T(0.5) * lam[c][0], T(0.5) * lam[c][1], T(0.5) * mu[b][0], T(0.5) * mu[b][1]};
      if (SIDE) {  // powers of two: exact
        r.ca0 *= w[c], r.ca1 *= w[c], r.cb0 *= w[b], r.cb1 *= w[b];
        r.la0 *= ga[c] * w[b], r.la1 *= gb[c] * w[b], r.mb0 *= ga[b] * w[c], r.mb1 *= gb[b] * w[c];
      }
      const O2Vals<T> n{u[nb[c][0]], u[nb[c][1]], u[nb[b][0]], u[nb[b][1]],
                        v[nb[c][0] + nb[b][0]], v[nb[c][0] + nb[b][1]], v[nb[c][1] + nb[b][0]], v[nb[c][1] + nb[b][1]]};
      const T uv = u[0], k = o2_row(r, uv, n);
      const long long pp = p + c * g.field;
      if (MODE == 3) {  // operator only
        f.u_next[pp] = k * (T(0.5) * irh);
        continue;
      }
      const T d = o2_delta<T, FORCED>(ks, k, kc, fr[c], dl[c]), un = o2_add(uv, d);
      if (MODE != STEP_LAST) {
        f.delta[pp] = d;
        f.u_next[pp] = un;
      }
      f.acc[pp] = o2_fma(T(s.wnew), un, MODE == STEP_FIRST ? o2_mul(T(s.w0), uv) : ap[c]);
    }
  };
  if (side)
    node(std::true_type{});
  else
    node(std::false_type{});
}

// ---------------------------------------------------------------------------
// Order 2, 3D: a CTA of 32 x 8 threads walks its columns of unknowns along z.
// u, lambda and mu of a plane (with a halo of one node) are staged in a ring of
// four planes (three in FP64, with a second barrier per plane); the next plane's
// loads are in flight while a plane is computed.  Nodes off the free sides take one formula
// without a test: a transposed centred difference needs no mask, because u
// vanishes on a Dirichlet plane and with it every difference along the plane.
// Warps with a node on a free side take the form with weights.
//
// 128^3 FP32: 122 -> 42 us per level (0.53 of the copy rate in the 72-byte count),
// 1740 -> 370 instructions a node; bound by shared-memory reads (59 a node) and by
// the barrier.  FP64, bound by its pipe: 1325 -> 475 us, 61^3 141 -> 62 us.  With
// every side free: 129 -> 61 us and 1481 -> 738 us.
// ---------------------------------------------------------------------------
constexpr int O2_TX = 32, O2_TY = 8, O2_SX = O2_TX + 2, O2_SY = O2_TY + 2, O2_PLANE = O2_SX * O2_SY;

// Planes per CTA: the walk of the busiest SM is shortest (two planes stand for a
// CTA's prologue).  21^3: 1, 61^3: 7, 128^3: 16 (FP32, at most 16: with 19, three CTAs an SM
// for four, 51 us for 42) or 19 (FP64).  At a fixed 16, 61^3 took 17 us in FP32 and 138
// in FP64 for 8.5 and 62, 21^3 17 and 176 for 2.6 and 13.
inline int o2_planes(int tiles, int nz, int most) {
  int best = 1;
  long long cost = 1LL << 62;
  for (int zc = 1; zc <= most && zc <= nz; ++zc) {
    const long long ctas = (long long)tiles * ((nz + zc - 1) / zc), c = (ctas + 151) / 152 * (zc + 2);
    if (c < cost) cost = c, best = zc;
  }
  return best;
}

// 2 h^2 rho M^{-1} K u at the node v of the middle plane: five fields (u, v, w,
// lambda, mu) O2_PLANE apart, dm and dp the ways to planes z - 1 and z + 1.  SIDE:
// the node may lie on a free side (lo, hi).  There a difference takes the node itself
// for the neighbour that is missing, over half the width (w = 2), which also drops
// that edge's pure term; the transposed difference weighs its two members by ga, gb
// (G(-1) - G(1) inside, 2 G(-1) + 2 G(0) and -2 G(0) - 2 G(1) at the ends).
template <typename T, bool SIDE>
__device__ __forceinline__ void o2_node(const T* v, int dm, int dp, const bool lo[3], const bool hi[3], T k[3]) {
  constexpr int F = O2_PLANE;
  int nb[3][2] = {{-1, 1}, {-O2_SX, O2_SX}, {dm, dp}};
  T w[3], ga[3], gb[3];
  if (SIDE) {
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      w[a] = lo[a] || hi[a] ? T(2) : T(1);
      ga[a] = lo[a] ? T(-2) : w[a];
      gb[a] = hi[a] ? T(-2) : w[a];
      if (lo[a]) nb[a][0] = 0;
      if (hi[a]) nb[a][1] = 0;
    }
  }
  const T l0 = v[3 * F], m0 = v[4 * F], p0 = l0 + T(2) * m0;
  T lam[3][2], mu[3][2];
#pragma unroll
  for (int a = 0; a < 3; ++a)
#pragma unroll
    for (int e = 0; e < 2; ++e) lam[a][e] = v[3 * F + nb[a][e]], mu[a][e] = v[4 * F + nb[a][e]];
  T pure[3];
#pragma unroll
  for (int al = 0; al < 3; ++al) {
    const T u0 = v[al * F];
    T t = T(0);
#pragma unroll
    for (int a = 0; a < 3; ++a) {  // edges along a: twice the mean coefficient
      const T cl = al == a ? p0 + (lam[a][0] + T(2) * mu[a][0]) : m0 + mu[a][0];
      const T cr = al == a ? p0 + (lam[a][1] + T(2) * mu[a][1]) : m0 + mu[a][1];
      const T dl = u0 - v[al * F + nb[a][0]], dr = u0 - v[al * F + nb[a][1]];
      if (SIDE) {
        t += w[a] * (cl * dl + cr * dr);
      } else {
        t += cl * dl;
        t += cr * dr;
      }
    }
    pure[al] = t;
  }
  if (SIDE) {
#pragma unroll
    for (int a = 0; a < 3; ++a) lam[a][0] *= ga[a], lam[a][1] *= gb[a], mu[a][0] *= ga[a], mu[a][1] *= gb[a];
  }
  T mixed[3] = {T(0), T(0), T(0)};  // four times the mixed terms
#pragma unroll
  for (int be = 0; be < 3; ++be)
#pragma unroll
    for (int al = 0; al < 3; ++al) {
      if (al == be) continue;
      // u_be at the four corners of the (al, be) square: (al side, be side)
      const T* const q = v + be * F;
      const T pp = q[nb[al][1] + nb[be][1]], pm = q[nb[al][1] + nb[be][0]];
      const T mp = q[nb[al][0] + nb[be][1]], mm = q[nb[al][0] + nb[be][0]];
      // Z_al(lambda C_be u_be) + Z_be(mu C_al u_be)
      T t = mixed[al];
      if (SIDE) {
        t += w[be] * (lam[al][0] * (mp - mm) - lam[al][1] * (pp - pm));
        t += w[al] * (mu[be][0] * (pm - mm) - mu[be][1] * (pp - mp));
      } else {
        t += lam[al][0] * (mp - mm);
        t -= lam[al][1] * (pp - pm);
        t += mu[be][0] * (pm - mm);
        t -= mu[be][1] * (pp - mp);
      }
      mixed[al] = t;
    }
#pragma unroll
  for (int al = 0; al < 3; ++al) k[al] = pure[al] + T(0.5) * mixed[al];
}

template <typename T, int MODE, bool FORCED>
__global__ void __launch_bounds__(O2_TX * O2_TY, sizeof(T) == 8 ? 2 : 4) step3d_o2(Geom g, WaveFields<T> f, StepScalars s, double kt2, int zc) {
  if (g.dim != 3) return;
  constexpr int R = sizeof(T) == 8 ? 3 : 4;
  __shared__ T ring[R][5 * O2_PLANE];
  const int t = threadIdx.y * O2_TX + threadIdx.x;
  const int nzc = (g.nu[2] + zc - 1) / zc;
  const int rhs = blockIdx.z / nzc;
  const int X0 = g.off[0] + (int)blockIdx.x * O2_TX, Y0 = g.off[1] + (int)blockIdx.y * O2_TY;
  const int z0 = g.off[2] + (int)(blockIdx.z % nzc) * zc, z1 = min(z0 + zc, g.off[2] + g.nu[2]);
  const long long ro = (long long)rhs * 3 * g.field;
  // the tile positions this thread brings in: two of the 34 x 10
  const int j0 = t, j1 = t + O2_TX * O2_TY;
  const bool two = j1 < O2_PLANE;
  const int q0 = (int)pidx(g, 0, 0, X0 - 1 + j0 % O2_SX, Y0 - 1 + j0 / O2_SX, 0);
  const int q1 = two ? (int)pidx(g, 0, 0, X0 - 1 + j1 % O2_SX, Y0 - 1 + j1 / O2_SX, 0) : q0;
  const int PL = (int)g.plane;
  const T* const U = f.u_cur + ro;
  T v[2][5];
  auto load = [&](int z) {
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      const int q = (e ? q1 : q0) + z * PL;
      if (e && !two) break;
#pragma unroll
      for (int c = 0; c < 3; ++c) v[e][c] = U[c * g.field + q];
      v[e][3] = __ldg(f.lam + q);
      v[e][4] = __ldg(f.mu + q);
    }
  };
  auto store = [&](int slot) {
    T* const r = ring[slot];
#pragma unroll
    for (int c = 0; c < 5; ++c) {
      r[c * O2_PLANE + j0] = v[0][c];
      if (two) r[c * O2_PLANE + j1] = v[1][c];
    }
  };
  pdl_wait();
  pdl_trigger();
  for (int z = z0 - 1; z <= z0 + 1; ++z) {  // z0 - 1 >= -1: ghost planes are zero
    load(z);
    store(z - z0 + 1);
  }
  int sa = 0, sb = 1, sc = 2;  // slots of planes z - 1, z, z + 1
  const int x = X0 + threadIdx.x, y = Y0 + threadIdx.y;
  const bool live = x < g.off[0] + g.nu[0] && y < g.off[1] + g.nu[1];
  // of the warp: one lane on a free side takes all of them through the general form
  const bool wside = __any_sync(0xffffffffu, live && (x == 0 || x == g.n[0] - 1 || y == 0 || y == g.n[1] - 1));
  const int o = (threadIdx.y + 1) * O2_SX + threadIdx.x + 1;
  const long long pc0 = pidx(g, 0, 0, x, y, 0);
  const T cs = T(kt2), fc = T(s.kt * s.cosn), w0 = T(s.w0), wnew = T(s.wnew);
  for (int z = z0; z < z1; ++z) {
    if (z + 1 < z1) load(z + 2);  // in flight during this plane
    const long long pc = pc0 + (long long)z * PL;
    T irh = T(0), dl[3], ap[3], fr[3];
    if (live) {
      irh = __ldg(f.irh2 + pc);
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        const long long p = ro + c * g.field + pc;
        dl[c] = (MODE == STEP_MID || MODE == STEP_LAST) ? f.delta[p] : T(0);
        ap[c] = (MODE == STEP_MID || MODE == STEP_LAST) ? f.acc[p] : T(0);
        fr[c] = FORCED ? __ldg(f.frho + p) : T(0);
      }
    }
    __syncthreads();  // plane z + 1 is in the ring; plane z - 2 is no longer read
    const bool side = wside || z == 0 || z == g.n[2] - 1;
    if (live) {
      const T* const b = ring[sb] + o;
      const int dm = (sa - sb) * (5 * O2_PLANE), dp = (sc - sb) * (5 * O2_PLANE);
      const bool lo[3] = {x == 0, y == 0, z == 0}, hi[3] = {x == g.n[0] - 1, y == g.n[1] - 1, z == g.n[2] - 1};
      T k[3];
      if (side)
        o2_node<T, true>(b, dm, dp, lo, hi, k);
      else
        o2_node<T, false>(b, dm, dp, lo, hi, k);
#pragma unroll
      for (int e = 0; e < 3; ++e) {
        const long long p = ro + e * g.field + pc;
        if (MODE == 3) {  // operator only
          f.u_next[p] = k[e] * (T(0.5) * irh);
          continue;
        }
        T ka = k[e] * (irh * cs);
        if (FORCED) ka += fc * fr[e];
        const T uv = b[e * O2_PLANE];
        const T d = MODE == STEP_FIRST ? T(-0.5) * ka : dl[e] - ka, un = uv + d;
        if (MODE != STEP_LAST) {
          f.delta[p] = d;
          f.u_next[p] = un;
        }
        f.acc[p] = MODE == STEP_FIRST ? w0 * uv + wnew * un : ap[e] + wnew * un;
      }
    }
    if (R == 3) __syncthreads();  // plane z - 1 is no longer read
    const int sn = R == 3 ? sa : (sc + 1) & 3;  // R = 4: the slot of plane z - 2
    if (z + 1 < z1) store(sn);
    sa = sb, sb = sc, sc = sn;
  }
}

// 12 times the interior difference: the order-4 kernels that carry the
// operator as 12 D (stresses 12 sigma, divergence 144 D sigma) apply the
// 1 / 144 once per node, with 1 / (rho h^2), instead of once per difference.
template <typename T>
__device__ __forceinline__ T c4u(T m2, T m1, T p1, T p2) {
  return m2 - T(8) * m1 + T(8) * p1 - p2;
}

// ---------------------------------------------------------------------------
// Order 4 (SBP), 3D: stress pass then divergence + update pass, the operator
// carried as 12 D (stress fields 12 sigma: xx, yy, zz, xy, xz, yz per rhs).
// A thread takes one node of a z plane, nodes numbered row after row without
// padding: no lane of a warp is idle at the end of a row (32 x 8 blocks left a fifth
// of them idle at 103 nodes).  Closure rows are four taps from a table by the
// node's class along an axis, for every lane of a warp alike.
//
// FP64 is bound by its pipe (2 lanes per clock and SM; 71 to 80% busy): 100
// FP64 instructions a node, against 159 with 1/12 in every difference and lanes of
// closure rows in branches of their own.  101 x 93 x 87 nodes: 265 -> 179 us per
// level, 64^3 122 -> 69 us, 110^3 384 -> 280 us.  FP32 (the z-march takes over above
// some 10^6 nodes): 64^3 29 -> 17 us.  Registers: 80 / 64 in FP64 for the stress and the
// divergence kernel (64 spill in the first), 64 in FP32.
// ---------------------------------------------------------------------------
constexpr int S3_THREADS = 256;

template <typename T>
struct S3Taps {  // 12 D per class: closure rows of the low side (0 .. 3), interior, of the high side (5 .. 8)
  int off[36];
  T w[36];
};

// class of line position p
__device__ __forceinline__ int s3_class(int p, int n) { return p < 4 ? p : (p > n - 5 ? 5 + (n - 1 - p) : 4); }

// 12 D at v along an axis of stride st, by the taps of class cls
template <typename T>
__device__ __forceinline__ T s3_taps12(const T* v, int st, int cls, const S3Taps<T>& t) {
  const int* o = t.off + 4 * cls;
  const T* w = t.w + 4 * cls;
  return w[0] * v[o[0] * st] + w[1] * v[o[1] * st] + w[2] * v[o[2] * st] + w[3] * v[o[3] * st];
}
template <typename T>
__device__ __forceinline__ T s3_c12(const T* v, int st) { return c4u(v[-2 * st], v[-st], v[st], v[2 * st]); }
// FP32: either form per axis (the compiler computes both and selects, which
// costs less than the registers of a second code path: 117 against 163 us per
// level at 128^3; in FP64, where an instruction costs forty issue slots, the second
// path pays: 203 against 286 us at 101 x 93 x 87)
template <typename T>
__device__ __forceinline__ T s3_either(const T* v, int st, bool taps, int cls, const S3Taps<T>& t) {
  return taps ? s3_taps12(v, st, cls, t) : s3_c12(v, st);
}

template <typename T>
__global__ void __launch_bounds__(S3_THREADS, sizeof(T) == 8 ? 3 : 4) sbp_stress3d(Geom g, const T* __restrict__ u, const T* __restrict__ lam,
                                                           const T* __restrict__ mu, T* __restrict__ sig,
                                                           const __grid_constant__ S3Taps<T> tp) {
  if (g.dim != 3) return;
  __shared__ S3Taps<T> st;
  if (threadIdx.x < 36) st.off[threadIdx.x] = tp.off[threadIdx.x], st.w[threadIdx.x] = tp.w[threadIdx.x];
  const int total = g.n[0] * g.n[1];
  const int i = blockIdx.x * S3_THREADS + threadIdx.x, ii = min(i, total - 1);
  const int y = ii / g.n[0], x = ii - y * g.n[0], z = blockIdx.y, rhs = blockIdx.z;
  const long long pc = pidx(g, 0, 0, x, y, z);
  const T l = lam[pc], m = mu[pc];  // static: read before the wait
  __syncthreads();
  pdl_wait();
  pdl_trigger();
  const int cx = s3_class(x, g.n[0]), cy = s3_class(y, g.n[1]), cz = s3_class(z, g.n[2]);
  const bool side = __any_sync(0xffffffffu, cx != 4 || cy != 4 || cz != 4);  // of the warp: no per-lane branch
  const int sy = g.np[0], sz = (int)g.plane;  // neighbour offsets: 5 planes index in 32 bits (checked at launch)
  const T* const U = u + (long long)rhs * 3 * g.field + pc;
  T d[3][3];
  if (sizeof(T) == 4) {
    const bool wx = __any_sync(0xffffffffu, cx != 4), wy = __any_sync(0xffffffffu, cy != 4), wz = cz != 4;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const T* b = U + c * g.field;
      d[c][0] = s3_either(b, 1, wx, cx, st);
      d[c][1] = s3_either(b, sy, wy, cy, st);
      d[c][2] = s3_either(b, sz, wz, cz, st);
    }
  } else if (!side) {
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const T* b = U + c * g.field;
      d[c][0] = s3_c12(b, 1);
      d[c][1] = s3_c12(b, sy);
      d[c][2] = s3_c12(b, sz);
    }
  } else {
#pragma unroll 1
    for (int c = 0; c < 3; ++c) {
      const T* b = U + c * g.field;
      const T e0 = s3_taps12(b, 1, cx, st), e1 = s3_taps12(b, sy, cy, st), e2 = s3_taps12(b, sz, cz, st);
      if (c == 0) d[0][0] = e0, d[0][1] = e1, d[0][2] = e2;
      else if (c == 1) d[1][0] = e0, d[1][1] = e1, d[1][2] = e2;
      else d[2][0] = e0, d[2][1] = e1, d[2][2] = e2;
    }
  }
  if (i >= total) return;
  const T ld = l * (d[0][0] + d[1][1] + d[2][2]), m2 = m + m;
  T* const o = sig + (long long)rhs * 6 * g.field + pc;
  const long long fld = g.field;
  o[0] = ld + m2 * d[0][0];
  o[fld] = ld + m2 * d[1][1];
  o[2 * fld] = ld + m2 * d[2][2];
  o[3 * fld] = m * (d[0][1] + d[1][0]);
  o[4 * fld] = m * (d[0][2] + d[2][0]);
  o[5 * fld] = m * (d[1][2] + d[2][1]);
}

template <typename T, int MODE, bool FORCED>
__global__ void __launch_bounds__(S3_THREADS, 4) sbp_div3d(Geom g, WaveFields<T> f, StepScalars s,
                                                           double kt144, double ktcos,
                                                           const __grid_constant__ S3Taps<T> tp) {
  if (g.dim != 3) return;
  __shared__ S3Taps<T> st;
  if (threadIdx.x < 36) st.off[threadIdx.x] = tp.off[threadIdx.x], st.w[threadIdx.x] = tp.w[threadIdx.x];
  const int total = g.nu[0] * g.nu[1];  // unknown nodes of the plane
  const int i = blockIdx.x * S3_THREADS + threadIdx.x, ii = min(i, total - 1);
  const int yi = ii / g.nu[0];
  const int x = ii - yi * g.nu[0] + g.off[0], y = yi + g.off[1], z = blockIdx.y + g.off[2], rhs = blockIdx.z;
  const long long pc = pidx(g, 0, 0, x, y, z);
  const T irh = f.irh2[pc];  // static: read before the wait
  __syncthreads();
  pdl_wait();
  pdl_trigger();
  const int cx = s3_class(x, g.n[0]), cy = s3_class(y, g.n[1]), cz = s3_class(z, g.n[2]);
  const bool side = __any_sync(0xffffffffu, cx != 4 || cy != 4 || cz != 4);
  const int sy = g.np[0], sz = (int)g.plane;
  const long long fld = g.field;
  const T* const S = f.sigma + (long long)rhs * 6 * fld + pc;  // planes xx, yy, zz, xy, xz, yz
  constexpr int row[3][3] = {{0, 3, 4}, {3, 1, 5}, {4, 5, 2}};
  T k[3];  // -144 h^2 rho M^{-1} K u
  const T bt = T(12.0 * 48.0 / 17.0);  // boundary terms of free sides: -D + H^{-1} B
  if (sizeof(T) == 4) {
    const bool wx = __any_sync(0xffffffffu, cx != 4), wy = __any_sync(0xffffffffu, cy != 4), wz = cz != 4;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const T* const a = S + row[c][0] * fld;
      const T* const b = S + row[c][1] * fld;
      const T* const e = S + row[c][2] * fld;
      k[c] = s3_either(a, 1, wx, cx, st) + s3_either(b, sy, wy, cy, st) + s3_either(e, sz, wz, cz, st);
      if (side) {
        if (x == 0) k[c] += bt * a[0];
        if (x == g.n[0] - 1) k[c] -= bt * a[0];
        if (y == 0) k[c] += bt * b[0];
        if (y == g.n[1] - 1) k[c] -= bt * b[0];
        if (z == 0) k[c] += bt * e[0];
        if (z == g.n[2] - 1) k[c] -= bt * e[0];
      }
    }
  } else if (!side) {
#pragma unroll
    for (int c = 0; c < 3; ++c)
      k[c] = s3_c12(S + row[c][0] * fld, 1) + s3_c12(S + row[c][1] * fld, sy) + s3_c12(S + row[c][2] * fld, sz);
  } else {
#pragma unroll 1
    for (int c = 0; c < 3; ++c) {
      const T* const a = S + (c == 0 ? 0 : c == 1 ? 3 : 4) * fld;
      const T* const b = S + (c == 0 ? 3 : c == 1 ? 1 : 5) * fld;
      const T* const e = S + (c == 0 ? 4 : c == 1 ? 5 : 2) * fld;
      T v = s3_taps12(a, 1, cx, st) + s3_taps12(b, sy, cy, st) + s3_taps12(e, sz, cz, st);
      if (x == 0) v += bt * a[0];
      if (x == g.n[0] - 1) v -= bt * a[0];
      if (y == 0) v += bt * b[0];
      if (y == g.n[1] - 1) v -= bt * b[0];
      if (z == 0) v += bt * e[0];
      if (z == g.n[2] - 1) v -= bt * e[0];
      if (c == 0) k[0] = v;
      else if (c == 1) k[1] = v;
      else k[2] = v;
    }
  }
  if (i >= total) return;
  const long long p0 = (long long)rhs * 3 * fld + pc;
  if (MODE == 3) {  // operator only
    const T a = irh * T(-1.0 / 144.0);
#pragma unroll
    for (int c = 0; c < 3; ++c) f.u_next[p0 + c * fld] = k[c] * a;
    return;
  }
  const T cs = irh * T(kt144), fc = T(ktcos);
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const long long p = p0 + c * fld;
    const T uv = f.u_cur[p];
    T d = MODE == STEP_FIRST ? k[c] * cs : f.delta[p] + k[c] * cs;
    if (FORCED) d -= fc * f.frho[p];
    if (MODE == STEP_FIRST) d *= T(0.5);
    const T un = uv + d;
    if (MODE != STEP_LAST) {
      f.delta[p] = d;
      f.u_next[p] = un;
    }
    f.acc[p] = MODE == STEP_FIRST ? T(s.w0) * uv + T(s.wnew) * un : f.acc[p] + T(s.wnew) * un;
  }
}

// ---------------------------------------------------------------------------
// Launchers
// ---------------------------------------------------------------------------
// Launch with programmatic stream serialization (see pdl_wait); EWH_PDL=0
// turns it off.
static bool pdl_enabled() {
  const char* e = getenv("EWH_PDL");
  return !(e && e[0] == '0');
}

template <typename... KArgs, typename... Args>
static cudaError_t launch_k(void (*kernel)(KArgs...), dim3 grid, dim3 block, cudaStream_t st, Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = 0;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = pdl_enabled() ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kernel, args...);
}

// 2D order-4 kernel variants (Geom::variant, chosen per context by the
// autotuner): 0 = stress + divergence pair (the only one in FP64), YM_VARIANT =
// the FP32 y-march (ewh_ymarch.cu).  EWH_STEP2D_O4=split|ym overrides it (read
// whenever launches are enqueued; a context captures its step graph once, on first use).
// ---------------------------------------------------------------------------
// Order 4 (SBP), 2D, in two launches: stresses, then divergence and update.  A
// thread takes 16 bytes' worth of nodes along x (four in FP32, two in FP64) of the
// rectangle where every difference is central and every node an unknown, with
// 16-byte loads (14 for the differences of four FP32 nodes instead of 64).
// Rectangle and frame (the nodes within some four of a side, one per thread, their
// closure rows as taps from a table) are numbered apart, so no warp runs both forms;
// the frame's blocks come first.  What no level writes is read before the wait for the
// previous kernel, and all loads precede the first store.  The operator is carried as
// 12 D (stresses 12 sigma, divergence 144 D sigma).
//
// Per level, against one node a thread in shared-memory tiles with six-tap closures: FP32
// 66^2 6.4 -> 3.6 us, 258^2 6.6 -> 3.9, 514^2 9.5 -> 6.1, 1026^2 22.6 -> 12.6, 2002^2
// 94 -> 59 us; FP64 66^2 10.1 -> 5.5, 1026^2 106 -> 87 us.  Small grids are bound by the two
// launches, FP32 by L2 and HBM (88 bytes a node and level; 2002^2: 0.88 of the copy
// rate), FP64 by its pipe.  One launch over tiles with recomputed stresses was slower
// at every size.
// ---------------------------------------------------------------------------
struct Part2d {
  int xa, ngx, nr;  // first column of the rectangle, its groups per row, its rows (from row 4)
  int nfc;          // frame columns in the rectangle's rows
  int nbf;          // blocks of frame nodes, in front
  int frame;        // frame nodes
};
constexpr int P2_THREADS = 64;

template <typename T>
struct Vec16;
template <>
struct Vec16<float> {
  using type = float4;
};
template <>
struct Vec16<double> {
  using type = double2;
};
// W vectors of 16 bytes at p (aligned), s elements apart
template <typename T, int W>
__device__ __forceinline__ void ld16(const T* p, T (*out)[16 / sizeof(T)], int s = 16 / sizeof(T)) {
#pragma unroll
  for (int k = 0; k < W; ++k)
    *reinterpret_cast<typename Vec16<T>::type*>(out[k]) = *reinterpret_cast<const typename Vec16<T>::type*>(p + k * s);
}
template <typename T>
__device__ __forceinline__ void st16(T* p, const T* v) {
  *reinterpret_cast<typename Vec16<T>::type*>(p) = *reinterpret_cast<const typename Vec16<T>::type*>(v);
}

// 12 D (central) of a group at v: along x from the 16 bytes before, at and
// after it, along y from the rows at -2, -1, 1 and 2.
template <typename T>
__device__ __forceinline__ void dx16(const T* v, T* d) {
  constexpr int V = 16 / sizeof(T);
  alignas(16) T w[3][V];
  ld16<T, 3>(v - V, w);
  const T* const c = &w[0][0] + V;
#pragma unroll
  for (int k = 0; k < V; ++k) d[k] = c4u(c[k - 2], c[k - 1], c[k + 1], c[k + 2]);
}
template <typename T>
__device__ __forceinline__ void dy16(const T* v, int sy, T* d) {
  constexpr int V = 16 / sizeof(T);
  alignas(16) T lo[2][V], hi[2][V];
  ld16<T, 2>(v - 2 * sy, lo, sy);
  ld16<T, 2>(v + sy, hi, sy);
#pragma unroll
  for (int k = 0; k < V; ++k) d[k] = c4u(lo[0][k], lo[1][k], hi[0][k], hi[1][k]);
}

// Position of a thread: frame node (true) or first node of a group; x < 0: none.
__device__ __forceinline__ bool part2d_pos(const Geom& g, const Part2d& c, int V, int& x, int& y) {
  x = -1;
  if ((int)blockIdx.x < c.nbf) {
    int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= c.frame) return true;
    if (j < 8 * g.n[0]) {
      y = j / g.n[0];
      x = j - y * g.n[0];
      if (y >= 4) y += g.n[1] - 8;
    } else {
      j -= 8 * g.n[0];
      y = j / c.nfc;
      x = j - y * c.nfc;
      if (x >= c.xa) x += c.ngx * V;
      y += 4;
    }
    return true;
  }
  const int i = (blockIdx.x - c.nbf) * blockDim.x + threadIdx.x;
  if (i >= c.ngx * c.nr) return false;
  y = i / c.ngx;
  x = c.xa + (i - y * c.ngx) * V;
  y += 4;
  return false;
}

// The closure taps into shared memory (frame blocks; blockDim.x >= 32)
template <typename T>
__device__ __forceinline__ void load_taps(const S3Taps<T>& tp, S3Taps<T>& st) {
  for (int i = threadIdx.x; i < 36; i += blockDim.x) st.off[i] = tp.off[i], st.w[i] = tp.w[i];
  __syncthreads();
}

template <typename T>
__global__ void __launch_bounds__(P2_THREADS) sbp_stress2d(Geom g, Part2d cp, const T* __restrict__ u,
                                                           const T* __restrict__ lam, const T* __restrict__ mu,
                                                           T* __restrict__ sig, const __grid_constant__ S3Taps<T> tp) {
  if (g.dim != 2) return;
  constexpr int V = 16 / sizeof(T);
  int x, y;
  const bool frame = part2d_pos(g, cp, V, x, y);
  const int rhs = blockIdx.y;
  const long long pc = x < 0 ? 0 : pidx(g, 0, 0, x, y, 0);
  const T* const U = u + (long long)rhs * 2 * g.field + pc;
  T* const out = sig + (long long)rhs * 3 * g.field + pc;
  const int sy = g.np[0];
  if (frame) {
    __shared__ S3Taps<T> taps;
    load_taps(tp, taps);
    const T l = lam[pc], m = mu[pc];
    pdl_wait();
    pdl_trigger();
    if (x < 0) return;
    const T* const W = U + g.field;
    const int cx = s3_class(x, g.n[0]), cy = s3_class(y, g.n[1]);
    const T u_x = s3_taps12(U, 1, cx, taps), u_y = s3_taps12(U, sy, cy, taps);
    const T v_x = s3_taps12(W, 1, cx, taps), v_y = s3_taps12(W, sy, cy, taps);
    const T ld = l * (u_x + v_y);
    out[0] = ld + T(2) * m * u_x;
    out[g.field] = ld + T(2) * m * v_y;
    out[2 * g.field] = m * (u_y + v_x);
    return;
  }
  alignas(16) T l[1][V], m[1][V];
  if (x >= 0) ld16<T, 1>(lam + pc, l), ld16<T, 1>(mu + pc, m);
  pdl_wait();
  pdl_trigger();
  if (x < 0) return;
  T u_x[V], u_y[V], v_x[V], v_y[V];
  dx16(U, u_x);
  dx16(U + g.field, v_x);
  dy16(U, sy, u_y);
  dy16(U + g.field, sy, v_y);
  alignas(16) T o[3][V];
#pragma unroll
  for (int k = 0; k < V; ++k) {
    const T ld = l[0][k] * (u_x[k] + v_y[k]);
    o[0][k] = ld + T(2) * m[0][k] * u_x[k];
    o[1][k] = ld + T(2) * m[0][k] * v_y[k];
    o[2][k] = m[0][k] * (u_y[k] + v_x[k]);
  }
#pragma unroll
  for (int k = 0; k < 3; ++k) st16(out + k * g.field, o[k]);
}

// Leapfrog / filter update of one value, kd = -M^{-1} K u / irh in units of 1 / kts (dl, ac: delta^n and
// the filter's sum in, the new ones out); the operator alone: un = -kd kts irh.  The value
// meets kts, then irh: M^{-1} K u alone exceeds the field by 1 / (c dt^2), and the product of
// the two constants would be one more rounding that every level of a node shares.
template <typename T, int MODE, bool FORCED>
__device__ __forceinline__ void pair_update(T kd, T kts, T irh, T fc, T fr, T w0, T wnew, T uv, T& dl, T& ac, T& un) {
  const T k = kd * kts;
  if (MODE == 3) {
    un = -k * irh;
    return;
  }
  T d = MODE == STEP_FIRST ? k * irh : dl + k * irh;
  if (FORCED) d -= fr * fc;
  if (MODE == STEP_FIRST) d *= T(0.5);
  un = uv + d;
  ac = MODE == STEP_FIRST ? w0 * uv + wnew * un : ac + wnew * un;
  dl = d;
}

// Divergence and update of both kinds of grid: component c from the fields at qc (along
// x) and rc (along y).  kts: c dt^2 (for the operator alone: 1) over the scale that the
// fields and the differences carry.  ktcos: c dt^2 cos(w t_n).
template <typename T, int MODE, bool FORCED>
__device__ __forceinline__ void div2d_part(const Geom& g, const Part2d& cp, const WaveFields<T>& f, const StepScalars& s,
                                           const S3Taps<T>& tp, int nf, int qu, int ru, int qv, int rv, double kts,
                                           double ktcos) {
  constexpr int V = 16 / sizeof(T);
  constexpr bool RD = MODE == STEP_MID || MODE == STEP_LAST;
  int x, y;
  const bool frame = part2d_pos(g, cp, V, x, y);
  const int rhs = blockIdx.y;
  const long long pc = x < 0 ? 0 : pidx(g, 0, 0, x, y, 0);
  const long long p0 = (long long)rhs * 2 * g.field + pc;
  const T* const sg = f.sigma + (long long)rhs * nf * g.field + pc;
  const T *const fqu = sg + qu * g.field, *const fru = sg + ru * g.field;
  const T *const fqv = sg + qv * g.field, *const frv = sg + rv * g.field;
  const int sy = g.np[0];
  if (frame) {
    __shared__ S3Taps<T> taps;
    load_taps(tp, taps);
    const bool unk = x >= 0 && is_unknown(g, x, y, 0);
    const T irh = f.irh2[pc];
    const T fr0 = FORCED ? f.frho[p0] : T(0), fr1 = FORCED ? f.frho[p0 + g.field] : T(0);
    pdl_wait();
    pdl_trigger();
    if (!unk) return;
    const T u0 = f.u_cur[p0], u1 = f.u_cur[p0 + g.field];
    T d0 = RD ? f.delta[p0] : T(0), d1 = RD ? f.delta[p0 + g.field] : T(0);
    T a0 = RD ? f.acc[p0] : T(0), a1 = RD ? f.acc[p0 + g.field] : T(0);
    const int cx = s3_class(x, g.n[0]), cy = s3_class(y, g.n[1]);
    const T ih = T(12.0 * 48.0 / 17.0);
    const T bx = x == 0 ? ih : (x == g.n[0] - 1 ? -ih : T(0)), by = y == 0 ? ih : (y == g.n[1] - 1 ? -ih : T(0));
    const T ku = s3_taps12(fqu, 1, cx, taps) + s3_taps12(fru, sy, cy, taps) + (bx * fqu[0] + by * fru[0]);
    const T kv = s3_taps12(fqv, 1, cx, taps) + s3_taps12(frv, sy, cy, taps) + (bx * fqv[0] + by * frv[0]);
    T n0, n1;
    pair_update<T, MODE, FORCED>(ku, T(kts), irh, T(ktcos), fr0, T(s.w0), T(s.wnew), u0, d0, a0, n0);
    pair_update<T, MODE, FORCED>(kv, T(kts), irh, T(ktcos), fr1, T(s.w0), T(s.wnew), u1, d1, a1, n1);
    if (MODE != STEP_LAST) f.u_next[p0] = n0, f.u_next[p0 + g.field] = n1;
    if (MODE == STEP_FIRST || MODE == STEP_MID) f.delta[p0] = d0, f.delta[p0 + g.field] = d1;
    if (MODE != 3) f.acc[p0] = a0, f.acc[p0 + g.field] = a1;
    return;
  }
  alignas(16) T irh[1][V], fr[2][V];
  if (x >= 0) {
    ld16<T, 1>(f.irh2 + pc, irh);
    if (FORCED) ld16<T, 1>(f.frho + p0, fr), ld16<T, 1>(f.frho + p0 + g.field, fr + 1);
  }
  pdl_wait();
  pdl_trigger();
  if (x < 0) return;
  alignas(16) T uv[2][V], dl[2][V], ac[2][V], dq[2][V], dr[2][V];
#pragma unroll
  for (int c = 0; c < 2; ++c) {  // all loads before the first store
    const long long p = p0 + c * g.field;
    ld16<T, 1>(f.u_cur + p, uv + c);
    if (RD) ld16<T, 1>(f.delta + p, dl + c), ld16<T, 1>(f.acc + p, ac + c);
    dx16(c ? fqv : fqu, dq[c]);
    dy16(c ? frv : fru, sy, dr[c]);
  }
#pragma unroll
  for (int c = 0; c < 2; ++c) {
    const long long p = p0 + c * g.field;
    alignas(16) T un[V];
#pragma unroll
    for (int k = 0; k < V; ++k) {
      pair_update<T, MODE, FORCED>(dq[c][k] + dr[c][k], T(kts), irh[0][k], T(ktcos), FORCED ? fr[c][k] : T(0), T(s.w0),
                                   T(s.wnew), uv[c][k], dl[c][k], ac[c][k], un[k]);
    }
    if (MODE != STEP_LAST) st16(f.u_next + p, un);
    if (MODE == STEP_FIRST || MODE == STEP_MID) st16(f.delta + p, dl[c]);
    if (MODE != 3) st16(f.acc + p, ac[c]);
  }
}

// stresses xx, yy, xy (12 sigma)
template <typename T, int MODE, bool FORCED>
__global__ void __launch_bounds__(P2_THREADS) sbp_div2d(Geom g, Part2d cp, WaveFields<T> f, StepScalars s,
                                                        double kts, double ktcos,
                                                        const __grid_constant__ S3Taps<T> tp) {
  if (g.dim != 2) return;
  div2d_part<T, MODE, FORCED>(g, cp, f, s, tp, 3, 0, 2, 2, 1, kts, ktcos);
}

// ---------------------------------------------------------------------------
// Order 4 (SBP), 2D, curvilinear grid (Section 4.1, curvilinear form): the
// node grid is the image of (q, r) = (i h, j h) under a smooth mapping.  The
// stress kernel forms physical derivatives from the SBP derivatives in q and
// r, u_x = (y_r u_q - y_q u_r) / J, u_y = (x_q u_r - x_r u_q) / J, the
// stresses (the 1/J rides on lambda / J and mu / J, which the context stores
// in place of lambda and mu), and the four J-weighted fluxes
//   F^q_u = y_r s_xx - x_r s_xy,  F^r_u = -y_q s_xx + x_q s_xy,
//   F^q_v = y_r s_xy - x_r s_yy,  F^r_v = -y_q s_xy + x_q s_yy;
// the divergence kernel forms -D_q F^q - D_r F^r + H^{-1} B F (the Cartesian
// kernel with the fluxes in place of the stresses) times 1/(rho J h^2).
// The metric planes are (y_r, -x_r, -y_q, x_q).
//
// In two kernels (see the 2D pair above), the differences divided by 12 at once.
// Per level, stress and divergence: 1026 x 1026 nodes 21.9 -> 14.6 us in FP32 (122 MB,
// mostly out of L2), 144 -> 131 us in FP64 (its pipe); 66 x 66 7.2 -> 3.6 us and 11.3 -> 7.1
// us.  A fused form (u, metrics and fluxes of a tile in shared memory) took 6.9 us at
// 66^2 and 38 us at 1026^2 in FP32.
// ---------------------------------------------------------------------------
template <typename T>
__device__ __forceinline__ void curv_flux(T uq, T ur, T vq, T vr, T a0, T a1, T a2, T a3, T l, T m, T* o0, T* o1, T* o2,
                                          T* o3) {
  const T u_x = a0 * uq + a2 * ur, u_y = a1 * uq + a3 * ur;  // J times the physical gradient
  const T v_x = a0 * vq + a2 * vr, v_y = a1 * vq + a3 * vr;
  const T div = u_x + v_y;
  const T sxx = l * div + T(2) * m * u_x, syy = l * div + T(2) * m * v_y, sxy = m * (u_y + v_x);
  *o0 = a0 * sxx + a1 * sxy;
  *o1 = a2 * sxx + a3 * sxy;
  *o2 = a0 * sxy + a1 * syy;
  *o3 = a2 * sxy + a3 * syy;
}

template <typename T>
__global__ void __launch_bounds__(P2_THREADS) curv_stress2d(Geom g, Part2d cp, const T* __restrict__ u,
                                                              const T* __restrict__ lam, const T* __restrict__ mu,
                                                              const T* __restrict__ met, T* __restrict__ sig,
                                                              const __grid_constant__ S3Taps<T> tp) {
  if (g.dim != 2) return;
  constexpr int V = 16 / sizeof(T);
  int x, y;
  const bool frame = part2d_pos(g, cp, V, x, y);
  const int rhs = blockIdx.y;
  const long long pc = x < 0 ? 0 : pidx(g, 0, 0, x, y, 0);  // lam, mu: lambda / J, mu / J
  const T* const U = u + (long long)rhs * 2 * g.field + pc;
  T* const out = sig + (long long)rhs * 4 * g.field + pc;
  if (frame) {
    __shared__ S3Taps<T> taps;
    load_taps(tp, taps);
    const T l = lam[pc], m = mu[pc], a0 = met[pc], a1 = met[g.field + pc], a2 = met[2 * g.field + pc];
    const T a3 = met[3 * g.field + pc];
    pdl_wait();
    pdl_trigger();
    if (x < 0) return;
    const T* const Vv = U + g.field;
    const int sy = g.np[0], cx = s3_class(x, g.n[0]), cy = s3_class(y, g.n[1]);
    const T w = T(1.0 / 12.0);
    const T uq = w * s3_taps12(U, 1, cx, taps), ur = w * s3_taps12(U, sy, cy, taps);
    const T vq = w * s3_taps12(Vv, 1, cx, taps), vr = w * s3_taps12(Vv, sy, cy, taps);
    curv_flux(uq, ur, vq, vr, a0, a1, a2, a3, l, m, out, out + g.field, out + 2 * g.field, out + 3 * g.field);
    return;
  }
  alignas(16) T a[4][V], l[1][V], m[1][V];
  if (x >= 0) {
#pragma unroll
    for (int k = 0; k < 4; ++k) ld16<T, 1>(met + k * g.field + pc, a + k);
    ld16<T, 1>(lam + pc, l);
    ld16<T, 1>(mu + pc, m);
  }
  pdl_wait();
  pdl_trigger();
  if (x < 0) return;
  const int sy = g.np[0];
  T uq[V], ur[V], vq[V], vr[V];
  dx16(U, uq);
  dx16(U + g.field, vq);
  dy16(U, sy, ur);
  dy16(U + g.field, sy, vr);
  alignas(16) T o[4][V];
  const T w = T(1.0 / 12.0);
#pragma unroll
  for (int k = 0; k < V; ++k)
    curv_flux(w * uq[k], w * ur[k], w * vq[k], w * vr[k], a[0][k], a[1][k], a[2][k], a[3][k], l[0][k], m[0][k], &o[0][k], &o[1][k],
              &o[2][k], &o[3][k]);
#pragma unroll
  for (int k = 0; k < 4; ++k) st16(out + k * g.field, o[k]);
}

// fluxes F^q_u, F^r_u, F^q_v, F^r_v; irh2 = 1 / (rho J h^2)
template <typename T, int MODE, bool FORCED>
__global__ void __launch_bounds__(P2_THREADS) curv_div2d(Geom g, Part2d cp, WaveFields<T> f, StepScalars s,
                                                         double kts, double ktcos,
                                                         const __grid_constant__ S3Taps<T> tp) {
  if (g.dim != 2) return;
  div2d_part<T, MODE, FORCED>(g, cp, f, s, tp, 4, 0, 1, 2, 3, kts, ktcos);
}

// Metric terms of a mapped grid (FP64, dense C-order planes, x fastest):
// x_q, x_r, y_q, y_r from the SBP first derivative over the node spacing h,
// J = x_q y_r - x_r y_q; out holds the planes (y_r, -x_r, -y_q, x_q, 1/J, J).
__global__ void curv_metrics_kernel(int n0, int n1, double h, const double* __restrict__ X,
                                    const double* __restrict__ Y, double* __restrict__ out) {
  const long long total = (long long)n0 * n1;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total;
       i += (long long)gridDim.x * blockDim.x) {
    const int x = (int)(i % n0), y = (int)(i / n0);
    const double xq = sbp_d1<double>(X + i, 1, x, n0) / h, xr = sbp_d1<double>(X + i, n0, y, n1) / h;
    const double yq = sbp_d1<double>(Y + i, 1, x, n0) / h, yr = sbp_d1<double>(Y + i, n0, y, n1) / h;
    const double J = xq * yr - xr * yq;
    out[i] = yr;
    out[total + i] = -xr;
    out[2 * total + i] = -yq;
    out[3 * total + i] = xq;
    out[4 * total + i] = 1.0 / J;
    out[5 * total + i] = J;
  }
}

cudaError_t launch_curv_metrics(int n0, int n1, double h, const double* X, const double* Y, double* out,
                                cudaStream_t st) {
  const long long total = (long long)n0 * n1;
  const int blocks = (int)std::min<long long>((total + 255) / 256, 4096);
  curv_metrics_kernel<<<blocks, 256, 0, st>>>(n0, n1, h, X, Y, out);
  return cudaGetLastError();
}

// The taps of 12 D per class (see S3Taps).
template <typename T>
static const S3Taps<T>& s3_taps() {
  static const S3Taps<T> t = [] {
    static const int cols[4][4] = {{0, 1, 2, 3}, {0, 2, -1, -1}, {0, 1, 3, 4}, {0, 2, 4, 5}};
    static const int in_off[4] = {-2, -1, 1, 2};
    static const double in_w[4] = {1.0, -8.0, 8.0, -1.0};
    S3Taps<T> q;
    for (int c = 0; c < 9; ++c)
      for (int k = 0; k < 4; ++k) {
        const int r = c < 4 ? c : c - 5, j = c == 4 ? 0 : cols[r][k];
        q.off[4 * c + k] = c == 4 ? in_off[k] : (j < 0 ? 0 : (c < 4 ? j - r : r - j));
        q.w[4 * c + k] = (T)(c == 4 ? in_w[k] : (j < 0 ? 0.0 : (c < 4 ? 12.0 : -12.0) * SBP_CLOSURE[r][j]));
      }
    return q;
  }();
  return t;
}

// Rectangle and frame of the 2D pair, and its launch shape.
template <typename T>
static Part2d part2d(const Geom& g, dim3* grd, dim3* blk) {
  constexpr int V = 16 / sizeof(T);
  Part2d cp;
  cp.xa = 4 + (V - (4 + g.padx) % V) % V;
  cp.nr = g.n[1] - 8;
  cp.ngx = cp.nr > 0 ? std::max(0, (g.n[0] - 4 - cp.xa) / V) : 0;
  cp.nfc = g.n[0] - V * cp.ngx;
  cp.frame = 8 * g.n[0] + cp.nfc * cp.nr;
  // blocks of 64 threads (mapped, 1026^2 FP32: 14.6 us a level, with 256 14.9, with 32 19.0), of
  // one warp where those would leave SMs short (202^2 FP64: 8.9 us, with 64 12.0)
  const int nt = (long long)(cp.frame + cp.ngx * cp.nr) * g.nrhs < 4LL * 152 * P2_THREADS ? 32 : P2_THREADS;
  cp.nbf = (cp.frame + nt - 1) / nt;
  *blk = dim3(nt);
  *grd = dim3(cp.nbf + (cp.ngx * cp.nr + nt - 1) / nt, g.nrhs);
  return cp;
}

template <typename T, int MODE, bool FORCED>
static cudaError_t launch_mode(const Geom& g, int order, const WaveFields<T>& f, const StepScalars& s,
                               cudaStream_t st, long long* nl) {
  if (order == 2) {
    if (g.dim == 2) {
      // tile height chosen per context (autotuner): 0 -> 8, 1 -> 4, 2 -> 16 rows
      const int ty = g.variant == 1 ? 4 : (g.variant == 2 ? 16 : 8);
      dim3 blk(32, ty), grd((g.nu[0] + 31) / 32, (g.nu[1] + ty - 1) / ty, g.nrhs);
      cudaError_t e = ty == 4    ? launch_k(step2d_o2<T, MODE, FORCED, 4>, grd, blk, st, g, f, s)
                      : ty == 16 ? launch_k(step2d_o2<T, MODE, FORCED, 16>, grd, blk, st, g, f, s)
                                 : launch_k(step2d_o2<T, MODE, FORCED, 8>, grd, blk, st, g, f, s);
      if (e != cudaSuccess) return e;
    } else {
      const int tx = (g.nu[0] + O2_TX - 1) / O2_TX, ty = (g.nu[1] + O2_TY - 1) / O2_TY;
      const int zc = o2_planes(tx * ty * g.nrhs, g.nu[2], sizeof(T) == 8 ? 32 : 16);
      dim3 blk(O2_TX, O2_TY), grd(tx, ty, (g.nu[2] + zc - 1) / zc * g.nrhs);
      cudaError_t e = launch_k(step3d_o2<T, MODE, FORCED>, grd, blk, st, g, f, s, 0.5 * s.kt, zc);
      if (e != cudaSuccess) return e;
    }
    if (nl) *nl += 1;
    return cudaGetLastError();
  }
  if (g.mapped) {  // curvilinear 2D order 4: stress + divergence
    dim3 grd, blk;
    const Part2d cp = part2d<T>(g, &grd, &blk);
    cudaError_t e = launch_k(curv_stress2d<T>, grd, blk, st, g, cp, (const T*)f.u_cur, f.lam, f.mu, f.met, f.sigma,
                             s3_taps<T>());
    if (e != cudaSuccess) return e;
    e = launch_k(curv_div2d<T, MODE, FORCED>, grd, blk, st, g, cp, f, s, (MODE == 3 ? 1.0 : s.kt) / 12.0, s.kt * s.cosn,
                 s3_taps<T>());
    if (e != cudaSuccess) return e;
    if (nl) *nl += 2;
    return cudaGetLastError();
  }
  if constexpr (sizeof(T) == 4 && MODE != 3) {
    // fused y-march: autotuner variant YM_VARIANT; EWH_STEP2D_O4=ym forces it
    const char* ev = getenv("EWH_STEP2D_O4");
    const bool ym = ev ? strcmp(ev, "ym") == 0 : g.variant == YM_VARIANT;
    if (g.dim == 2 && ym && f.zm && f.zm->ok[0]) {
      cudaError_t e = launch_ymarch(g, *f.zm, f, (StepMode)MODE, s, st);
      if (e != cudaSuccess) return e;
      if (nl) *nl += 1;
      return cudaGetLastError();
    }
  }
  if (g.dim == 2) {
    dim3 grd, blk;
    const Part2d cp = part2d<T>(g, &grd, &blk);
    cudaError_t e = launch_k(sbp_stress2d<T>, grd, blk, st, g, cp, (const T*)f.u_cur, f.lam, f.mu, f.sigma, s3_taps<T>());
    if (e != cudaSuccess) return e;
    e = launch_k(sbp_div2d<T, MODE, FORCED>, grd, blk, st, g, cp, f, s, (MODE == 3 ? 1.0 : s.kt) / 144.0, s.kt * s.cosn,
                 s3_taps<T>());
    if (e != cudaSuccess) return e;
  } else {
    if constexpr (sizeof(T) == 4 && MODE != 3) {
      // fused z-march: autotuner variants 1 (64 x 8 tiles) and 2 (32 x 8);
      // EWH_STEP3D_O4=pair|zm16|zm8 (zm16: 64 x 8, else 32 x 8) overrides it
      const char* ev = getenv("EWH_STEP3D_O4");
      int zk = g.variant == 1 ? 0 : (g.variant == 2 ? 1 : -1);
      if (ev) zk = ev[0] != 'z' ? -1 : (strcmp(ev, "zm16") == 0 ? 0 : 1);
      if (zk >= 0 && f.zm && f.zm->ok[zk]) {
        cudaError_t e = launch_zmarch(g, *f.zm, zk, f, (StepMode)MODE, s, st);
        if (e != cudaSuccess) return e;
        if (nl) *nl += 1;
        return cudaGetLastError();
      }
    }
    if (5 * g.plane >= (1LL << 31) || (long long)g.n[0] * g.n[1] >= (1LL << 31) - S3_THREADS) return cudaErrorInvalidValue;
    const S3Taps<T>& tp = s3_taps<T>();
    auto blocks = [](long long n) { return (unsigned)((n + S3_THREADS - 1) / S3_THREADS); };
    cudaError_t e = launch_k(sbp_stress3d<T>, dim3(blocks((long long)g.n[0] * g.n[1]), g.n[2], g.nrhs), dim3(S3_THREADS),
                             st, g, (const T*)f.u_cur, f.lam, f.mu, f.sigma, tp);
    if (e != cudaSuccess) return e;
    e = launch_k(sbp_div3d<T, MODE, FORCED>, dim3(blocks((long long)g.nu[0] * g.nu[1]), g.nu[2], g.nrhs), dim3(S3_THREADS),
                 st, g, f, s, s.kt / 144.0, s.kt * s.cosn, tp);
    if (e != cudaSuccess) return e;
  }
  if (nl) *nl += 2;
  return cudaGetLastError();
}

template <typename T>
cudaError_t launch_step(const Geom& g, int order, const WaveFields<T>& f, StepMode mode,
                        const StepScalars& s, cudaStream_t st, long long* nl) {
  const bool forced = f.frho != nullptr;
  switch (mode) {
    case STEP_FIRST:
      return forced ? launch_mode<T, STEP_FIRST, true>(g, order, f, s, st, nl)
                    : launch_mode<T, STEP_FIRST, false>(g, order, f, s, st, nl);
    case STEP_MID:
      return forced ? launch_mode<T, STEP_MID, true>(g, order, f, s, st, nl)
                    : launch_mode<T, STEP_MID, false>(g, order, f, s, st, nl);
    default:
      return forced ? launch_mode<T, STEP_LAST, true>(g, order, f, s, st, nl)
                    : launch_mode<T, STEP_LAST, false>(g, order, f, s, st, nl);
  }
}

template <typename T>
cudaError_t launch_minvK(const Geom& g, int order, const T* u, T* out, const T* lam, const T* mu,
                         const T* irh2, T* sigma, cudaStream_t st, long long* nl, const T* met) {
  WaveFields<T> f{};
  f.met = met;
  f.u_cur = const_cast<T*>(u);
  f.u_next = out;
  f.lam = lam;
  f.mu = mu;
  f.irh2 = irh2;
  f.frho = nullptr;
  f.sigma = sigma;
  StepScalars s{};
  return launch_mode<T, 3, false>(g, order, f, s, st, nl);
}

// ---------------------------------------------------------------------------
// Order 4 (SBP), 2D, FP32: every time level of a wave solve in ONE
// cooperative launch per group of right-hand sides, with the state held on
// chip.
//
// One CTA of NT threads per SM owns a wx x wy block of nodes of one
// right-hand side (every block at least 8 x 8, so SBP closure reaches stay
// inside the halos); a launch holds px x py blocks of each of rg right-hand
// sides, and the groups of a multi-rhs context run one launch after another.  Its nodes
// on central rows and columns (x, y in [4, n - 5]) form a rectangle, done in
// pairs along x with no per-node test; the others (within 4 nodes of a side:
// SBP closures, boundary terms, Dirichlet nodes) are special and take a pass
// of their own with the general code.  The CTA keeps
//   in shared memory: u on the block +- 4 nodes, the stresses on the block
//                     +- 2 nodes, delta on the block, the special nodes'
//                     filter accumulators;
//   in registers:     the filter accumulators of its regular node pairs
//                     (pair t + NT k of the rectangle for thread t, k < NP).
// Per time level a CTA reloads only the 4-node halo ring of u (its
// neighbours' rims, written at the previous level to a global exchange
// buffer), recomputes the stresses on block +- 2 from u on block +- 4, forms
// -D sigma + H^{-1} B sigma and the leapfrog/filter update of its own nodes
// (same arithmetic as the split kernels), writes its own 4-node rim to the
// other exchange buffer and counts itself in at a grid barrier; the central
// stresses of the next level that need no halo are computed before it waits
// there.  One barrier per level; lambda, mu, 1/(rho h^2) (and f/rho) are the
// only other global reads.  Barrier waits are bounded in time; on a timeout
// the kernel raises an error flag, every CTA leaves at its next barrier and
// fills its accumulator nodes with NaN, which the solve reports as a
// breakdown.
// ---------------------------------------------------------------------------
constexpr int RS_HU = 4;  // u halo
constexpr int RS_HS = 2;  // stress halo

__device__ __forceinline__ unsigned ld_acquire_gpu(const unsigned* p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ unsigned long long global_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// Grid barrier pieces: a release add to count a CTA in, acquire loads to
// poll (see rs_arrive / rs_wait).
__device__ __forceinline__ void red_release_gpu(unsigned* p, unsigned v) {
  asm volatile("red.release.gpu.global.add.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}


// Split form of the grid barrier: rs_arrive after a __syncthreads that
// orders the CTA's writes (thread 0 counts the CTA in with a release add);
// rs_wait polls until `target` CTAs have arrived (each wait bounded: it gives
// up after `lim` ns or 2^22 polls, or when another CTA raised the error flag,
// which it then sees every 256 polls; a zero limit gives up at once, without
// polling) and ends with a __syncthreads.  Work that needs none of the other
// CTAs' data goes between the two.
__device__ __forceinline__ void rs_arrive(unsigned* bar) {
  if (threadIdx.x == 0) red_release_gpu(bar, 1u);
}

// Raise the error flag; the CTA that raises it first counts the launch in
// bar[4].  Returns 0 (the wait failed).
__device__ __forceinline__ int rs_give_up(unsigned* bar) {
  if (atomicExch(bar + 1, 1u) == 0u) atomicAdd(bar + 4, 1u);
  return 0;
}

__device__ __forceinline__ bool rs_wait(unsigned* bar, unsigned target, int* s_ok, unsigned long long lim) {
  if (threadIdx.x == 0) {
    int ok = ld_acquire_gpu(bar + 1) == 0u;
    if (ok && lim == 0ull) ok = rs_give_up(bar);
    const unsigned long long t0 = global_ns();
    for (unsigned spins = 1; ok && ld_acquire_gpu(bar) < target; ++spins) {
      if ((spins & 255u) == 0u) {
        if (ld_acquire_gpu(bar + 1) != 0u) {
          ok = 0;
        } else if (spins > (1u << 22) || global_ns() - t0 > lim) {
          ok = rs_give_up(bar);
        }
      }
    }
    *s_ok = ok;
  }
  __syncthreads();
  return *s_ok != 0;
}

__device__ __forceinline__ bool rs_closure(int x, int n) { return x < 4 || x > n - 5; }

struct ResidentShape {
  int px, bx, by, ex;  // CTAs along x; interior block width; block height; first block width
  int nb;              // CTAs per right-hand side (px * py): CTA b holds block b % nb of rhs b / nb
};

// The shared-memory layout is fixed at compile time (so every stencil and
// plane offset is an immediate): blocks are at most RS_BXMAX x RS_BYMAX nodes.
constexpr int RS_BXMAX = 132;
constexpr int RS_BYMAX = 54;
constexpr int RS_UX = RS_BXMAX + 2 * RS_HU;  // u tile row stride
constexpr int RS_SX = RS_BXMAX + 2 * RS_HS;  // stress tile row stride
constexpr int RS_UPLANE = (RS_BYMAX + 2 * RS_HU) * RS_UX;
constexpr int RS_SPLANE = (RS_BYMAX + 2 * RS_HS) * RS_SX;
constexpr int RS_DPLANE = RS_BYMAX * RS_BXMAX;
constexpr int RS_OFF_V = RS_UPLANE;              // u, component 1
constexpr int RS_OFF_XX = 2 * RS_UPLANE;         // stresses xx, yy, xy
constexpr int RS_OFF_YY = RS_OFF_XX + RS_SPLANE;
constexpr int RS_OFF_XY = RS_OFF_YY + RS_SPLANE;
constexpr int RS_OFF_DU = RS_OFF_XY + RS_SPLANE;  // delta, components 0 and 1
constexpr int RS_OFF_DV = RS_OFF_DU + RS_DPLANE;
constexpr int RS_OFF_TAB = RS_OFF_DV + RS_DPLANE;  // copy of the SBP closure rows (4 x 6)
extern __shared__ float rs_smem[];  // dynamic shared memory of the resident kernel

// Own nodes on an SBP closure row or column (within 4 nodes of a side of the
// grid) are updated in a pass of their own; their filter accumulators live
// here (2 per node, at most RS_SPECIAL_MAX nodes per block).
constexpr int RS_SPECIAL_MAX = 1400;
constexpr int RS_OFF_SACC = RS_OFF_TAB + 24;
constexpr int RS_FLOATS = RS_OFF_SACC + 2 * RS_SPECIAL_MAX;

// Position j of the part of a W x H region outside the rectangle
// [x0, x1) x [y0, y1) (which may be empty: then y0 = H): rows [0, y0), rows
// [y1, H), then columns [0, x0) and [x1, W) of the rows between.  It has
// W H - (x1 - x0)(y1 - y0) positions.
__device__ __forceinline__ void rs_frame_pos(int j, int W, int H, int x0, int x1, int y0, int y1, int& x, int& y) {
  const int top = y0 * W;
  if (j < top) {
    y = j / W;
    x = j - y * W;
    return;
  }
  j -= top;
  const int bot = (H - y1) * W;
  if (j < bot) {
    const int r = j / W;
    y = y1 + r;
    x = j - r * W;
    return;
  }
  j -= bot;
  const int sw = x0 + (W - x1);
  const int r = j / sw, c = j - r * sw;
  y = y0 + r;
  x = c < x0 ? c : x1 + (c - x0);
}

// SBP first derivative as sbp_d1, with the closure rows read from the shared
// copy `tab`: lanes on different closure rows then read different banks
// instead of serialising on the constant cache.
__device__ __forceinline__ float rs_sbp_d1(const float* v, int s, int p, int N, const float* tab) {
  if (p < 4) {
    float acc = 0.f;
#pragma unroll
    for (int j = 0; j < 6; ++j) acc += tab[p * 6 + j] * v[(j - p) * s];
    return acc;
  }
  if (p > N - 5) {
    const int r = N - 1 - p;
    float acc = 0.f;
#pragma unroll
    for (int j = 0; j < 6; ++j) acc -= tab[r * 6 + j] * v[(r - j) * s];
    return acc;
  }
  return (v[-2 * s] - 8.0f * v[-s] + 8.0f * v[s] - v[2 * s]) * (1.0f / 12.0f);
}

// Advance a thread's position in a w-wide row-major walk by (sx, sy) = the
// thread count split into whole rows and a remainder.
__device__ __forceinline__ void walk_next(int& x, int& y, int w, int sx, int sy) {
  x += sx;
  y += sy;
  if (x >= w) {
    x -= w;
    ++y;
  }
}

// Stresses at one stress-tile position (qx, qy) of the block at (X0, Y0):
// the general form (SBP closures; nothing outside the grid).
__device__ __forceinline__ void rs_stress_gen(const float* __restrict__ lam, const float* __restrict__ mu, int n0,
                                              int n1, int npx, int X0, int Y0, int obase, int qx, int qy,
                                              const float* tab) {
  const int x = X0 + qx - RS_HS, y = Y0 + qy - RS_HS;
  if (x < 0 || x >= n0 || y < 0 || y >= n1) return;
  const int o = obase + (qy - RS_HS) * npx + (qx - RS_HS);
  const float l = __ldg(lam + o), m = __ldg(mu + o);
  const int pu = (qy + RS_HU - RS_HS) * RS_UX + (qx + RS_HU - RS_HS);
  const float* U = rs_smem + pu;
  const float* V = rs_smem + RS_OFF_V + pu;
  float u_x, v_x, u_y, v_y;
  if (x < 4 || x > n0 - 5) {
    u_x = rs_sbp_d1(U, 1, x, n0, tab);
    v_x = rs_sbp_d1(V, 1, x, n0, tab);
  } else {
    u_x = c4(U[-2], U[-1], U[1], U[2]);
    v_x = c4(V[-2], V[-1], V[1], V[2]);
  }
  if (y < 4 || y > n1 - 5) {
    u_y = rs_sbp_d1(U, RS_UX, y, n1, tab);
    v_y = rs_sbp_d1(V, RS_UX, y, n1, tab);
  } else {
    u_y = c4(U[-2 * RS_UX], U[-RS_UX], U[RS_UX], U[2 * RS_UX]);
    v_y = c4(V[-2 * RS_UX], V[-RS_UX], V[RS_UX], V[2 * RS_UX]);
  }
  const float div = u_x + v_y;
  const int ps = qy * RS_SX + qx;
  rs_smem[RS_OFF_XX + ps] = l * div + 2.0f * m * u_x;
  rs_smem[RS_OFF_YY + ps] = l * div + 2.0f * m * v_y;
  rs_smem[RS_OFF_XY + ps] = m * (u_y + v_x);
}

// Stresses at the central positions (qx, qy) and (qx + 1, qy), qx even,
// with 8-byte shared accesses (every plane offset and row stride is even).
__device__ __forceinline__ void rs_stress_pair(const float* __restrict__ lam, const float* __restrict__ mu, int npx,
                                               int obase, int qx, int qy) {
  const int o = obase + (qy - RS_HS) * npx + (qx - RS_HS);
  const float l0 = __ldg(lam + o), l1 = __ldg(lam + o + 1);
  const float m0 = __ldg(mu + o), m1 = __ldg(mu + o + 1);
  const int pu = (qy + RS_HU - RS_HS) * RS_UX + (qx + RS_HU - RS_HS);  // even
  const float2* U = reinterpret_cast<const float2*>(rs_smem + pu);
  const float2* V = reinterpret_cast<const float2*>(rs_smem + RS_OFF_V + pu);
  constexpr int RU = RS_UX / 2;
  const float2 ua = U[-1], ub = U[0], uc = U[1];
  const float2 va = V[-1], vb = V[0], vc = V[1];
  const float ux0 = c4(ua.x, ua.y, ub.y, uc.x), ux1 = c4(ua.y, ub.x, uc.x, uc.y);
  const float vx0 = c4(va.x, va.y, vb.y, vc.x), vx1 = c4(va.y, vb.x, vc.x, vc.y);
  const float2 um2 = U[-2 * RU], um1 = U[-RU], up1 = U[RU], up2 = U[2 * RU];
  const float2 vm2 = V[-2 * RU], vm1 = V[-RU], vp1 = V[RU], vp2 = V[2 * RU];
  const float uy0 = c4(um2.x, um1.x, up1.x, up2.x), uy1 = c4(um2.y, um1.y, up1.y, up2.y);
  const float vy0 = c4(vm2.x, vm1.x, vp1.x, vp2.x), vy1 = c4(vm2.y, vm1.y, vp1.y, vp2.y);
  const float div0 = ux0 + vy0, div1 = ux1 + vy1;
  const int ps = qy * RS_SX + qx;  // even
  *reinterpret_cast<float2*>(rs_smem + RS_OFF_XX + ps) =
      make_float2(l0 * div0 + 2.0f * m0 * ux0, l1 * div1 + 2.0f * m1 * ux1);
  *reinterpret_cast<float2*>(rs_smem + RS_OFF_YY + ps) =
      make_float2(l0 * div0 + 2.0f * m0 * vy0, l1 * div1 + 2.0f * m1 * vy1);
  *reinterpret_cast<float2*>(rs_smem + RS_OFF_XY + ps) = make_float2(m0 * (uy0 + vx0), m1 * (uy1 + vx1));
}

// Per-level scalars of the leapfrog/filter update.
struct RsLevel {
  float kt, w0, wnew, cosn;
  int first;  // level 0: Taylor start
  int last;   // last level: u^{n+1} is not stored
};

// -D sigma + H^{-1} B sigma at own node (ix, iy), times 1/(rho h^2), plus the
// forcing: the general form (SBP closures, boundary terms).
__device__ __forceinline__ void rs_accel_gen(const Geom& g, const float* __restrict__ irh2,
                                             const float* __restrict__ frho, int F, int X0, int Y0, int obase, int ix,
                                             int iy, const RsLevel& L, const float* tab, float& au, float& av) {
  const int n0 = g.n[0], n1 = g.n[1];
  const int x = X0 + ix, y = Y0 + iy;
  const int ps = (iy + RS_HS) * RS_SX + (ix + RS_HS);
  const float* Sxx = rs_smem + RS_OFF_XX + ps;
  const float* Syy = rs_smem + RS_OFF_YY + ps;
  const float* Sxy = rs_smem + RS_OFF_XY + ps;
  float kxu, kxv, kyu, kyv;
  if (x < 4 || x > n0 - 5) {
    kxu = rs_sbp_d1(Sxx, 1, x, n0, tab);
    kxv = rs_sbp_d1(Sxy, 1, x, n0, tab);
  } else {
    kxu = c4(Sxx[-2], Sxx[-1], Sxx[1], Sxx[2]);
    kxv = c4(Sxy[-2], Sxy[-1], Sxy[1], Sxy[2]);
  }
  if (y < 4 || y > n1 - 5) {
    kyu = rs_sbp_d1(Sxy, RS_SX, y, n1, tab);
    kyv = rs_sbp_d1(Syy, RS_SX, y, n1, tab);
  } else {
    kyu = c4(Sxy[-2 * RS_SX], Sxy[-RS_SX], Sxy[RS_SX], Sxy[2 * RS_SX]);
    kyv = c4(Syy[-2 * RS_SX], Syy[-RS_SX], Syy[RS_SX], Syy[2 * RS_SX]);
  }
  float ku = -kxu - kyu;
  float kv = -kxv - kyv;
  const float inv_h0 = 48.0f / 17.0f;
  if (x == 0) {
    ku -= inv_h0 * Sxx[0];
    kv -= inv_h0 * Sxy[0];
  } else if (x == n0 - 1) {
    ku += inv_h0 * Sxx[0];
    kv += inv_h0 * Sxy[0];
  }
  if (y == 0) {
    ku -= inv_h0 * Sxy[0];
    kv -= inv_h0 * Syy[0];
  } else if (y == n1 - 1) {
    ku += inv_h0 * Sxy[0];
    kv += inv_h0 * Syy[0];
  }
  const int o = obase + iy * g.np[0] + ix;
  const float irh = __ldg(irh2 + o);
  au = ku * irh;
  av = kv * irh;
  if (frho) {
    au += __ldg(frho + o) * L.cosn;
    av += __ldg(frho + F + o) * L.cosn;
  }
}

// Leapfrog/filter update of own node (ix, iy) from its accelerations (the
// arithmetic of leapfrog_update in FP32): delta and u in shared memory, the
// accumulators in acu, acv.
__device__ __forceinline__ void rs_update(int ix, int iy, float au, float av, const RsLevel& L, float& acu,
                                          float& acv) {
  const int pu = (iy + RS_HU) * RS_UX + (ix + RS_HU);
  const int pd = iy * RS_BXMAX + ix;
  const float uu = rs_smem[pu], uv = rs_smem[RS_OFF_V + pu];
  float du, dv;
  if (L.first) {
    du = -0.5f * L.kt * au;
    dv = -0.5f * L.kt * av;
  } else {
    du = rs_smem[RS_OFF_DU + pd] - L.kt * au;
    dv = rs_smem[RS_OFF_DV + pd] - L.kt * av;
  }
  const float nu_ = uu + du, nv_ = uv + dv;
  if (L.first) {
    acu = L.w0 * uu + L.wnew * nu_;
    acv = L.w0 * uv + L.wnew * nv_;
  } else {
    acu += L.wnew * nu_;
    acv += L.wnew * nv_;
  }
  rs_smem[RS_OFF_DU + pd] = du;
  rs_smem[RS_OFF_DV + pd] = dv;
  if (!L.last) {
    rs_smem[pu] = nu_;
    rs_smem[RS_OFF_V + pu] = nv_;
  }
}

template <int NT, int NP>
__global__ void __launch_bounds__(NT, 1) step2d_o4_resident(Geom g, ResidentShape sh, ResidentIO iop) {
  if (g.dim != 2) return;
  __shared__ int s_ok;
  const unsigned long long wait_ns = *reinterpret_cast<const unsigned long long*>(iop.bar + 2);
  const int n0 = g.n[0], n1 = g.n[1];
  // this CTA's right-hand side (of the launch's group) and block
  const int rloc = blockIdx.x / sh.nb, bid = blockIdx.x - rloc * sh.nb;
  ResidentIO io = iop;
  {
    const long long ro = (long long)rloc * 2 * g.field;
    io.u0 += ro;
    io.xbuf0 += ro;
    io.xbuf1 += ro;
    io.acc += ro;
    if (io.frho) io.frho += ro;
  }
  const int cx = bid % sh.px;
  const int X0 = cx == 0 ? 0 : sh.ex + (cx - 1) * sh.bx, Y0 = (bid / sh.px) * sh.by;
  const int wx = cx == 0 ? sh.ex : min(sh.bx, n0 - X0), wy = min(sh.by, n1 - Y0);
  // u: [RS_BYMAX + 8][RS_UX] per component, block node (0, 0) at (4, 4);
  // stresses: [RS_BYMAX + 4][RS_SX], block node (0, 0) at (2, 2);
  // delta of the own nodes: [RS_BYMAX][RS_BXMAX]
  float* const su = rs_smem;
  float* const sv = rs_smem + RS_OFF_V;
  float* const sxx = rs_smem + RS_OFF_XX;
  float* const syy = rs_smem + RS_OFF_YY;
  float* const sxy = rs_smem + RS_OFF_XY;
  float* const tab = rs_smem + RS_OFF_TAB;
  float* const sacc = rs_smem + RS_OFF_SACC;
  const int t = threadIdx.x;
  const int F = (int)g.field;  // < 2^31 (checked at creation)
  const int npx = g.np[0];
  const int obase = (Y0 + PAD) * npx + X0 + g.padx;     // padded offset of block node (0, 0)
  const int ubase = obase - RS_HU * npx - RS_HU;         // ... of u tile position (0, 0)
  const int ux = wx + 2 * RS_HU, uy = wy + 2 * RS_HU;
  const int sxn = wx + 2 * RS_HS, syn = wy + 2 * RS_HS;
  // Stress positions on central rows and columns (x and y in [4, n - 5]):
  // the rectangle [qa, qb) x [ra, rb) of the stress tile; the rest (closure
  // rows and columns, positions outside the grid) is the stress frame.
  int qa = max(0, 6 - X0), qb = min(sxn, n0 - 2 - X0), ra = max(0, 6 - Y0), rb = min(syn, n1 - 2 - Y0);
  if (qb <= qa || rb <= ra) qa = qb = 0, ra = rb = syn;
  qb = qa + ((qb - qa) & ~1);  // even width: the rectangle is done in pairs of positions
  if (qb == qa) ra = rb = syn;
  const int wq = qb - qa, nsframe = sxn * syn - wq * (rb - ra);
  // Of the central positions, those whose stencil reads only the own u (tile
  // columns and rows [4, w + 4)): [ia, ib) x [ja, jb), even width, computed
  // while the other CTAs finish the previous level.  In pair columns of the
  // central rectangle: [pa, pb) x [ja, jb); the rest of the rectangle (the
  // outer pairs) follows the halo ring.
  int ia = max(qa, 4), ib = min(qb, wx), ja = max(ra, 4), jb = min(rb, wy);
  ib = ib > ia ? ia + ((ib - ia) & ~1) : ia;
  const int wp = wq >> 1;
  int pa = (ia - qa) >> 1, pb = (ib - qa) >> 1, pja = ja - ra, pjb = jb - ra;
  if (pb <= pa || pjb <= pja) pa = pb = 0, pja = pjb = rb - ra;
  const int wpi = pb - pa, nouter = wp * (rb - ra) - wpi * (pjb - pja);
  // Own nodes on central rows and columns: the rectangle [xa, xb) x [ya, yb)
  // of the block (all unknowns, no closure, no boundary term); the others
  // (within 4 nodes of a side of the grid) are the special nodes.
  int xa = max(0, 4 - X0), xb = min(wx, n0 - 4 - X0), ya = max(0, 4 - Y0), yb = min(wy, n1 - 4 - Y0);
  if (xb <= xa || yb <= ya) xa = xb = 0, ya = yb = wy;
  xb = xa + ((xb - xa) & ~1);  // even width: regular nodes are updated in pairs
  if (xb == xa) ya = yb = wy;
  const int wr = xb - xa, nreg = wr * (yb - ya), nspec = wx * wy - nreg;
  const int wr2 = wr >> 1, npair = nreg >> 1;
  if (t < 24) tab[t] = c_sbp_f[t / 6][t % 6];

  {  // u^0 on the whole tile
    int lx = t % ux, ly = t / ux;
    const int rx = NT % ux, ry = NT / ux;
    for (; ly < uy; walk_next(lx, ly, ux, rx, ry)) {
      const int o = ubase + ly * npx + lx;
      su[ly * RS_UX + lx] = __ldcg(io.u0 + o);
      sv[ly * RS_UX + lx] = __ldcg(io.u0 + F + o);
    }
  }
  // walk of this thread's regular node pairs: l = t + NT k -> (xa + 2 (l % wr2), ya + l / wr2);
  // (ip, iy) below are relative to (xa / 2, ya)
  const int wrs = max(wr2, 1);
  const int ix0 = t % wrs, iy0 = t / wrs;
  const int qstep = NT / wrs, rstep = NT % wrs;
  float ac0[NP], ac1[NP], ac2[NP], ac3[NP];  // u, v of the pair's first node; u, v of its second
#pragma unroll
  for (int k = 0; k < NP; ++k) ac0[k] = ac1[k] = ac2[k] = ac3[k] = 0.f;
  RsLevel L;
  L.kt = (float)io.kt;
  L.w0 = (float)io.w0;
  bool alive = true;
  __syncthreads();

  for (int n = 0;; ++n) {
    if (wpi > 0) {  // central stresses that need only the own u, in pairs
      int pp = t % wpi, qy = ja + t / wpi;
      const int rx = NT % wpi, ry = NT / wpi;
      for (; qy < jb; walk_next(pp, qy, wpi, rx, ry))
        rs_stress_pair(io.lam, io.mu, npx, obase, qa + 2 * (pa + pp), qy);
    }
    if (n > 0) {
      if (!rs_wait(io.bar, (unsigned)n * gridDim.x, &s_ok, wait_ns)) {
        alive = false;
        break;
      }
      // halo ring of u^n from the neighbours' rims
      const float* xbuf = (n & 1) ? io.xbuf1 : io.xbuf0;
      {  // top and bottom strips: tile rows 0..3 and wy+4..wy+7, all columns
        int lx = t % ux, r = t / ux;
        const int rx = NT % ux, ry = NT / ux;
        for (; r < 2 * RS_HU; walk_next(lx, r, ux, rx, ry)) {
          const int ly = r < RS_HU ? r : wy + r;
          const int o = ubase + ly * npx + lx;
          su[ly * RS_UX + lx] = __ldcg(xbuf + o);
          sv[ly * RS_UX + lx] = __ldcg(xbuf + F + o);
        }
      }
      for (int i = t; i < 2 * RS_HU * wy; i += NT) {  // side strips: columns 0..3 and wx+4..wx+7
        const int c = i & (2 * RS_HU - 1), ly = RS_HU + (i >> 3);
        const int lx = c < RS_HU ? c : wx + c;
        const int o = ubase + ly * npx + lx;
        su[ly * RS_UX + lx] = __ldcg(xbuf + o);
        sv[ly * RS_UX + lx] = __ldcg(xbuf + F + o);
      }
    }
    __syncthreads();
    for (int j = t; j < nouter; j += NT) {  // the outer central pairs
      int pc, r;
      rs_frame_pos(j, wp, rb - ra, pa, pb, pja, pjb, pc, r);
      rs_stress_pair(io.lam, io.mu, npx, obase, qa + 2 * pc, ra + r);
    }
    for (int j = t; j < nsframe; j += NT) {  // the stress frame: general form
      int qx, qy;
      rs_frame_pos(j, sxn, syn, qa, qb, ra, rb, qx, qy);
      rs_stress_gen(io.lam, io.mu, n0, n1, npx, X0, Y0, obase, qx, qy, tab);
    }
    __syncthreads();
    // divergence and leapfrog/filter update of the own nodes
    L.first = n == 0;
    L.last = n == io.nsteps - 1;
    L.cosn = (float)io.cosn[n];
    L.wnew = (float)io.wnew[n];
    float* xo = (n & 1) ? io.xbuf0 : io.xbuf1;  // rims of u^{n+1}
    int ix = ix0, iy = iy0;
#pragma unroll
    for (int k = 0; k < NP; ++k) {  // regular node pairs: central differences only
      if (t + k * NT < npair) {
        const int jx = xa + 2 * ix, jy = ya + iy;
        const int ps = (jy + RS_HS) * RS_SX + (jx + RS_HS);  // even
        const float2* SXX = reinterpret_cast<const float2*>(sxx + ps);
        const float2* SYY = reinterpret_cast<const float2*>(syy + ps);
        const float2* SXY = reinterpret_cast<const float2*>(sxy + ps);
        constexpr int RS2 = RS_SX / 2;
        const float2 xa_ = SXX[-1], xb_ = SXX[0], xc_ = SXX[1];
        const float2 ya_ = SXY[-1], yb_ = SXY[0], yc_ = SXY[1];
        const float kxu0 = c4(xa_.x, xa_.y, xb_.y, xc_.x), kxu1 = c4(xa_.y, xb_.x, xc_.x, xc_.y);
        const float kxv0 = c4(ya_.x, ya_.y, yb_.y, yc_.x), kxv1 = c4(ya_.y, yb_.x, yc_.x, yc_.y);
        const float2 sm2 = SXY[-2 * RS2], sm1 = SXY[-RS2], sp1 = SXY[RS2], sp2 = SXY[2 * RS2];
        const float2 tm2 = SYY[-2 * RS2], tm1 = SYY[-RS2], tp1 = SYY[RS2], tp2 = SYY[2 * RS2];
        const float kyu0 = c4(sm2.x, sm1.x, sp1.x, sp2.x), kyu1 = c4(sm2.y, sm1.y, sp1.y, sp2.y);
        const float kyv0 = c4(tm2.x, tm1.x, tp1.x, tp2.x), kyv1 = c4(tm2.y, tm1.y, tp1.y, tp2.y);
        const float ku0 = -kxu0 - kyu0, ku1 = -kxu1 - kyu1;
        const float kv0 = -kxv0 - kyv0, kv1 = -kxv1 - kyv1;
        const int o = obase + jy * npx + jx;
        const float r0 = __ldg(io.irh2 + o), r1 = __ldg(io.irh2 + o + 1);
        float au0 = ku0 * r0, av0 = kv0 * r0, au1 = ku1 * r1, av1 = kv1 * r1;
        if (io.frho) {
          au0 += __ldg(io.frho + o) * L.cosn;
          au1 += __ldg(io.frho + o + 1) * L.cosn;
          av0 += __ldg(io.frho + F + o) * L.cosn;
          av1 += __ldg(io.frho + F + o + 1) * L.cosn;
        }
        const int pu = (jy + RS_HU) * RS_UX + (jx + RS_HU);  // even
        const int pd = jy * RS_BXMAX + jx;                   // even
        float2* Up = reinterpret_cast<float2*>(su + pu);
        float2* Vp = reinterpret_cast<float2*>(sv + pu);
        float2* Dup = reinterpret_cast<float2*>(rs_smem + RS_OFF_DU + pd);
        float2* Dvp = reinterpret_cast<float2*>(rs_smem + RS_OFF_DV + pd);
        const float2 uu = *Up, uv = *Vp;
        float2 du, dv;
        if (L.first) {
          du = make_float2(-0.5f * L.kt * au0, -0.5f * L.kt * au1);
          dv = make_float2(-0.5f * L.kt * av0, -0.5f * L.kt * av1);
        } else {
          const float2 d0 = *Dup, d1 = *Dvp;
          du = make_float2(d0.x - L.kt * au0, d0.y - L.kt * au1);
          dv = make_float2(d1.x - L.kt * av0, d1.y - L.kt * av1);
        }
        const float2 nu_ = make_float2(uu.x + du.x, uu.y + du.y), nv_ = make_float2(uv.x + dv.x, uv.y + dv.y);
        if (L.first) {
          ac0[k] = L.w0 * uu.x + L.wnew * nu_.x;
          ac1[k] = L.w0 * uv.x + L.wnew * nv_.x;
          ac2[k] = L.w0 * uu.y + L.wnew * nu_.y;
          ac3[k] = L.w0 * uv.y + L.wnew * nv_.y;
        } else {
          ac0[k] += L.wnew * nu_.x;
          ac1[k] += L.wnew * nv_.x;
          ac2[k] += L.wnew * nu_.y;
          ac3[k] += L.wnew * nv_.y;
        }
        *Dup = du;
        *Dvp = dv;
        if (!L.last) {
          *Up = nu_;
          *Vp = nv_;
          const bool rowrim = jy < RS_HU || jy >= wy - RS_HU;
          if (rowrim || jx < RS_HU || jx >= wx - RS_HU) {
            xo[o] = nu_.x;
            xo[F + o] = nv_.x;
          }
          if (rowrim || jx + 1 < RS_HU || jx + 1 >= wx - RS_HU) {
            xo[o + 1] = nu_.y;
            xo[F + o + 1] = nv_.y;
          }
        }
      }
      walk_next(ix, iy, wr2, rstep, qstep);
    }
    for (int j = t; j < nspec; j += NT) {  // special nodes: general form, accumulators in shared memory
      int jx, jy;
      rs_frame_pos(j, wx, wy, xa, xb, ya, yb, jx, jy);
      const int x = X0 + jx, y = Y0 + jy;
      const bool unk = (x > 0 || g.lo_free[0]) && (x < n0 - 1 || g.hi_free[0]) && (y > 0 || g.lo_free[1]) &&
                       (y < n1 - 1 || g.hi_free[1]);
      if (unk) {
        float au, av;
        rs_accel_gen(g, io.irh2, io.frho, F, X0, Y0, obase, jx, jy, L, tab, au, av);
        rs_update(jx, jy, au, av, L, sacc[2 * j], sacc[2 * j + 1]);
      }
      if (!L.last && (jx < RS_HU || jx >= wx - RS_HU || jy < RS_HU || jy >= wy - RS_HU)) {
        const int o = obase + jy * npx + jx;
        const int pu = (jy + RS_HU) * RS_UX + (jx + RS_HU);
        xo[o] = su[pu];
        xo[F + o] = sv[pu];
      }
    }
    if (L.last) break;
    __syncthreads();  // this level's u and rims are written
    rs_arrive(io.bar);
  }
  // accumulators of the own unknowns (NaN when the barrier gave up)
  const float nanv = __int_as_float(0x7fc00000);
  int ix = ix0, iy = iy0;
#pragma unroll
  for (int k = 0; k < NP; ++k) {
    if (t + k * NT < npair) {
      const int o = obase + (ya + iy) * npx + (xa + 2 * ix);
      io.acc[o] = alive ? ac0[k] : nanv;
      io.acc[F + o] = alive ? ac1[k] : nanv;
      io.acc[o + 1] = alive ? ac2[k] : nanv;
      io.acc[F + o + 1] = alive ? ac3[k] : nanv;
    }
    walk_next(ix, iy, wr2, rstep, qstep);
  }
  __syncthreads();  // the special accumulators were written by other threads
  for (int j = t; j < nspec; j += NT) {
    int jx, jy;
    rs_frame_pos(j, wx, wy, xa, xb, ya, yb, jx, jy);
    const int x = X0 + jx, y = Y0 + jy;
    if ((x > 0 || g.lo_free[0]) && (x < n0 - 1 || g.hi_free[0]) && (y > 0 || g.lo_free[1]) &&
        (y < n1 - 1 || g.hi_free[1])) {
      const int o = obase + jy * npx + jx;
      io.acc[o] = alive ? sacc[2 * j] : nanv;
      io.acc[F + o] = alive ? sacc[2 * j + 1] : nanv;
    }
  }
}

static size_t resident_smem() { return sizeof(float) * (size_t)RS_FLOATS; }

// Opt the kernel in to the device's largest dynamic shared memory (the same
// value for every context, so plans of different sizes never undo each
// other; set before any launch or capture) and report CTAs per SM at smem.
template <int NT, int NP>
static cudaError_t resident_prepare(int smem_max, size_t smem, int* per_sm) {
  cudaFuncAttributes fa;
  cudaError_t e = cudaFuncGetAttributes(&fa, step2d_o4_resident<NT, NP>);
  if (e != cudaSuccess) return e;
  const int dyn_max = smem_max - (int)fa.sharedSizeBytes;  // static + dynamic <= opt-in limit
  if ((long long)smem > dyn_max) return cudaErrorInvalidValue;
  e = cudaFuncSetAttribute(step2d_o4_resident<NT, NP>, cudaFuncAttributeMaxDynamicSharedMemorySize, dyn_max);
  if (e != cudaSuccess) return e;
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(per_sm, step2d_o4_resident<NT, NP>, NT, smem);
}

static cudaError_t resident_prepare_shape(int shape, int smem_max, size_t smem, int* per_sm) {
  switch (shape) {
    case 0: return resident_prepare<RS_SHAPE_THREADS[0], RS_SHAPE_PAIRS[0]>(smem_max, smem, per_sm);
    case 1: return resident_prepare<RS_SHAPE_THREADS[1], RS_SHAPE_PAIRS[1]>(smem_max, smem, per_sm);
    case 2: return resident_prepare<RS_SHAPE_THREADS[2], RS_SHAPE_PAIRS[2]>(smem_max, smem, per_sm);
    default: return cudaErrorInvalidValue;
  }
}

ResidentPlan plan_resident_o4(const Geom& g, int shape) {
  ResidentPlan best;
  if (g.dim != 2 || g.nrhs < 1 || g.field >= (1LL << 31) || shape < 0 || shape >= RS_SHAPES) return best;
  int dev = 0, sms = 0, smem_max = 0, coop = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&smem_max, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev) != cudaSuccess || !coop) {
    cudaGetLastError();
    return best;
  }
  // every CTA of a launch must be resident at once
  int per_sm = 0;
  const cudaError_t e = resident_prepare_shape(shape, smem_max, resident_smem(), &per_sm);
  const bool verbose = getenv("EWH_VERBOSE") != nullptr;
  if (e != cudaSuccess || per_sm < 1) {
    if (verbose) fprintf(stderr, "ewh: resident shape %d unusable (%s)\n", shape, cudaGetErrorString(e));
    cudaGetLastError();
    return best;
  }
  const int ctas = per_sm * sms;  // co-resident CTAs of one launch
  const int R = g.nrhs;
  const long long cap = 2LL * RS_SHAPE_THREADS[shape] * RS_SHAPE_PAIRS[shape];
  const int n0 = g.n[0], n1 = g.n[1];
  // Blocks that hold x-closure columns (the first and last along x) take
  // about RS_EDGE_COST longer per node (a few lanes of their warps diverge):
  // they get proportionally fewer columns, so all CTAs reach each barrier
  // together.
  constexpr double RS_EDGE_COST = 1.1;
  // A level costs a CTA about its tile work plus a fixed part (the barrier,
  // the halo exchange) worth RS_LEVEL_FIXED tile positions.  With several
  // right-hand sides, each launch carries a group of rg of them (rg x px x py
  // CTAs, all co-resident) and the groups run one after another: the cost is
  // the number of groups times the slowest CTA's level.
  constexpr double RS_LEVEL_FIXED = 3000.0;
  double best_cost = -1.0;
  for (int px = 1; px <= ctas && px <= n0 / 8; ++px) {
    int bx, ex, last;
    if (px == 1) {
      bx = ex = last = n0;
    } else {
      bx = px == 2 ? (n0 + 1) / 2 : (int)std::ceil(n0 / (px - 2 + 2.0 / RS_EDGE_COST));
      ex = px == 2 ? bx : (n0 - (px - 2) * bx) / 2;
      last = n0 - ex - (px - 2) * bx;
    }
    if (ex < 8 || last < 8 || bx > RS_BXMAX || ex > RS_BXMAX || last > RS_BXMAX) continue;
    const int wmax = std::max(bx, std::max(ex, last));
    for (int py = 1; px * py <= ctas && py <= n1 / 8; ++py) {
      const int by = (n1 + py - 1) / py;
      const int pya = (n1 + by - 1) / by;
      if (n1 - (pya - 1) * by < 8) continue;
      if ((long long)wmax * by > cap || by > RS_BYMAX) continue;
      // nodes within 4 of a side of the grid, per block, fit their shared accumulators
      auto spec = [&](int X0, int w, int Y0, int h) {
        const int a = std::max(0, 4 - X0), b0 = std::min(w, n0 - 4 - X0), b = b0 > a ? a + ((b0 - a) & ~1) : b0;
        const int c = std::max(0, 4 - Y0), d = std::min(h, n1 - 4 - Y0);
        return w * h - ((b > a && d > c) ? (b - a) * (d - c) : 0);
      };
      bool fits = true;
      for (int cy = 0; cy < pya && fits; ++cy)
        for (int cx = 0; cx < px && fits; ++cx) {
          const int X0 = cx == 0 ? 0 : ex + (cx - 1) * bx;
          const int w = cx == 0 ? ex : std::min(bx, n0 - X0);
          fits = spec(X0, w, cy * by, std::min(by, n1 - cy * by)) <= RS_SPECIAL_MAX;
        }
      if (!fits) continue;
      const size_t sm = resident_smem();
      if (sm > (size_t)smem_max) continue;
      // per-CTA work (u tile + stress tile) of the slowest block
      auto work = [&](int w) { return (double)(w + 2 * RS_HU) * (by + 2 * RS_HU) + (double)(w + 2 * RS_HS) * (by + 2 * RS_HS); };
      const double level = px == 1 ? work(bx) * RS_EDGE_COST
                                   : std::max(work(bx), RS_EDGE_COST * work(std::max(ex, last)));
      const int nb = px * pya;
      const int rg0 = std::min(R, ctas / nb);
      if (rg0 < 1) continue;
      const int groups = (R + rg0 - 1) / rg0;
      const double cost = groups * (level + RS_LEVEL_FIXED);
      if (best_cost < 0 || cost < best_cost) {
        best_cost = cost;
        best.ok = 1;
        best.shape = shape;
        best.px = px;
        best.py = pya;
        best.bx = bx;
        best.ex = ex;
        best.by = by;
        best.smem = sm;
        best.groups = groups;
        best.rg = (R + groups - 1) / groups;  // balanced groups
      }
    }
  }
  if (!best.ok) return best;
  if (verbose)
    fprintf(stderr,
            "ewh: resident shape %d: %d x %d CTAs of %d (first %d) x %d nodes per rhs, %d rhs per launch in %d "
            "launches, %zu B shared\n",
            shape, best.px, best.py, best.bx, best.ex, best.by, best.rg, best.groups, best.smem);
  return best;
}

template <int NT, int NP>
static cudaError_t resident_launch(const Geom& g, const ResidentPlan& p, const ResidentIO& io, int nr,
                                   cudaStream_t st) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(nr * p.px * p.py);
  cfg.blockDim = dim3(NT);
  cfg.dynamicSmemBytes = p.smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  ResidentShape sh{p.px, p.bx, p.by, p.ex, p.px * p.py};
  return cudaLaunchKernelEx(&cfg, step2d_o4_resident<NT, NP>, g, sh, io);
}

// The groups of right-hand sides one after another, each one cooperative
// launch (its barrier words zeroed first).
cudaError_t launch_resident_o4(const Geom& g, const ResidentPlan& p, const ResidentIO& io, cudaStream_t st) {
  if (!p.ok || g.dim != 2 || io.nsteps < 1 || p.rg < 1 || (long long)p.rg * p.groups < g.nrhs)
    return cudaErrorInvalidValue;
  for (int k = 0; k < p.groups; ++k) {
    const int r0 = k * p.rg, nr = std::min(p.rg, g.nrhs - r0);
    if (nr < 1) break;
    ResidentIO gi = io;
    const long long ro = (long long)r0 * 2 * g.field;
    gi.u0 += ro;
    gi.xbuf0 += ro;
    gi.xbuf1 += ro;
    gi.acc += ro;
    if (gi.frho) gi.frho += ro;
    cudaError_t e = cudaMemsetAsync(io.bar, 0, 2 * sizeof(unsigned), st);
    if (e != cudaSuccess) return e;
    switch (p.shape) {
      case 0: e = resident_launch<RS_SHAPE_THREADS[0], RS_SHAPE_PAIRS[0]>(g, p, gi, nr, st); break;
      case 1: e = resident_launch<RS_SHAPE_THREADS[1], RS_SHAPE_PAIRS[1]>(g, p, gi, nr, st); break;
      case 2: e = resident_launch<RS_SHAPE_THREADS[2], RS_SHAPE_PAIRS[2]>(g, p, gi, nr, st); break;
      default: return cudaErrorInvalidValue;
    }
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

template cudaError_t launch_step<float>(const Geom&, int, const WaveFields<float>&, StepMode,
                                        const StepScalars&, cudaStream_t, long long*);
template cudaError_t launch_step<double>(const Geom&, int, const WaveFields<double>&, StepMode,
                                         const StepScalars&, cudaStream_t, long long*);
template cudaError_t launch_minvK<float>(const Geom&, int, const float*, float*, const float*, const float*,
                                         const float*, float*, cudaStream_t, long long*, const float*);
template cudaError_t launch_minvK<double>(const Geom&, int, const double*, double*, const double*,
                                          const double*, const double*, double*, cudaStream_t, long long*,
                                          const double*);

}  // namespace ewh
