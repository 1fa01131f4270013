// Order 4 (SBP), 3D, FP32: one fused launch per leapfrog level that marches
// along z.  It computes the level of the time-corrected explicit scheme
// (Section 4.3, eq. elastic-time-explicit-corrected) in increment form with
// the trapezoid accumulation of eq. (qoper), for the order-4 operator
//   M^{-1} K u = (1 / (rho h^2)) sum_a [ -D_a sigma_{.a} + H_a^{-1} B_a sigma_{.a} ]
// (pointwise energy density with fourth-order diagonal-norm SBP first
// derivatives D; the stresses sigma = lambda div u I + mu (grad u + grad u^T)).
//
// Each CTA owns tiles of TX x 8 unknown columns (TX = 64: one CTA of 12 warps per
// SM, TX = 32: two of 6) and walks them plane by plane.  A thread holds a pair of
// nodes adjacent along x, computed with packed FP32 instructions.  Per plane s it
//   - waits for the u planes that the stresses of plane s read: bulk-tensor (TMA)
//     loads of the tile +- 4 nodes in x and y into a ring of 8 plane buffers, one
//     mbarrier each;
//   - forms the stresses, scaled by 12 (12 D from unscaled central differences or
//     12x closure rows), on the tile +- 2 nodes: the own rows by the own warps,
//     the rows above and below by the halo warps, the pairs to the left and right
//     by a second pass of the first of these; xx, yy, xy, xz, yz go into one of two
//     plane buffers, so that one barrier per plane is enough;
//   - after it forms the in-plane part of -D sigma + H^{-1} B sigma of the own
//     nodes and adds the plane's z stresses, still in registers, to the pending
//     sums of the outputs s - 2 .. s + 2 (the central difference along z, by
//     column instead of by row: four packed instructions per component and no
//     ring of stress planes);
//   - completes output plane s - 2 with the leapfrog/filter update (8-byte loads
//     and stores; the operands are requested ahead of the barrier).
// Only u^n, delta, acc, lambda, mu, 1/(rho h^2) (and f/rho) are read and only
// delta, u^{n+1} and acc written: the stresses never leave the chip, except for
// the six planes next to each z side, which the outputs on z closure rows (the
// first and last four) read back: every thread keeps its own column of them in
// the stress scratch field.
//
// 256^3: 571 us per level (0.31 of the copy rate in the 72-byte count), against
// 790 us with rings of z stresses and in-plane sums in shared memory.  Bound by
// latency: 12 warps of 168 registers per SM issue 0.33 instructions per clock and
// scheduler; 96 registers and 18 warps spill (815 us), and with the shared memory
// taken a spill goes to L2.
//
// The grid is persistent: the (rhs, tile, plane) work is split into equal
// contiguous shares, one per CTA, each a few (tile, z range) segments.
// Waits on the mbarriers are bounded (the wait limit of the context's control
// words): a CTA that gives up counts itself in ctl[4], fills the accumulator
// of its remaining outputs with NaN and returns.
#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <cstdio>
#include <cstdlib>
#include <cstring>

#include "ewh_internal.cuh"
#include "ewh_march.cuh"

namespace ewh {

namespace {

constexpr int ZM_RU = 8;  // u plane ring: planes s - 3 .. s + 3 of the current stress plane s, and one in flight
static_assert((ZM_RU & (ZM_RU - 1)) == 0, "ring index by mask");

template <int TX, int TY>
struct ZmLayout {
  static constexpr int PW = TX / 2;                  // pairs per row
  static constexpr int RPW = 32 / PW;                // rows per warp
  static constexpr int NWO = TY / RPW;               // warps of the own rows,
  static constexpr int NWY = 4 / RPW;                // of the 2 + 2 halo rows,
  static_assert(2 * TY <= 32, "the left and right halo pairs are one more pass of the first halo warp");
  static constexpr int NT = 32 * (NWO + NWY);
  static constexpr int UX = TX + 8, UY = TY + 8;     // u tile: x from X0 - 4 (the bulk-tensor box), y from Y0 - 4
  static constexpr int SX = TX + 4, SY = TY + 4;     // stress tile: from X0 - 2, Y0 - 2
  static constexpr int UPLANE = UX * UY;             // one component of one u plane (floats)
  static constexpr int USLOT = 3 * UPLANE;
  static constexpr int SPLANE = SX * SY;             // one in-plane stress component
  static constexpr int SBUF = 5 * SPLANE;            // xx, yy, xy, xz, yz; two buffers
  static constexpr int OFF_SIP = ZM_RU * USLOT;
  static constexpr int OFF_CLS = OFF_SIP + 2 * SBUF;        // tap offsets (int) then weights, per class
  static constexpr int FLOATS = OFF_CLS + 8 * ZM_CLASSES;   // even: the mbarriers follow, 8-byte aligned
  static constexpr size_t BYTES = 128 + sizeof(float) * FLOATS + sizeof(uint64_t) * ZM_RU;
  static constexpr unsigned TX_BYTES = sizeof(float) * USLOT;  // one bulk-tensor box
  static_assert(USLOT % 32 == 0, "u ring slots stay 128-byte aligned");
  static_assert(FLOATS % 2 == 0 && SBUF % 2 == 0 && UPLANE % 2 == 0, "8-byte pairs and mbarriers");
  static_assert(OFF_CLS % 4 == 0, "16-byte table rows");
};

struct ZmScalars {
  float kt144;      // c dt^2 / 144
  float w0, wnew;   // trapezoid weights of level 0 (first level only) and of the new level
  float fcos144;    // 144 cos(w t_n)
  float bt12;       // 12 * 48 / 17: the boundary term H^{-1} B in the scaled arithmetic
  int shx, shy;     // tile origins: off[a] - sh + tile size * k (see zm_shift)
  // 12 D at a node of class k as four taps: offsets toff[4 k ..] and weights
  // tcf[4 k ..] (classes 0..3: SBP rows 0..3 from the low side, 4: interior,
  // 5..8: rows 0..3 from the high side; zero weights pad the short rows)
  int toff[4 * ZM_CLASSES];
  float tcf[4 * ZM_CLASSES];
};

// ---- pairs: two FP32 values per instruction ----------------------------------
__device__ __forceinline__ uint64_t p2(float2 v) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(v.x), "f"(v.y));
  return r;
}
__device__ __forceinline__ float2 f2(uint64_t v) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
  return r;
}
__device__ __forceinline__ float2 add2(float2 a, float2 b) {
  uint64_t r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(p2(a)), "l"(p2(b)));
  return f2(r);
}
__device__ __forceinline__ float2 mul2(float2 a, float2 b) {
  uint64_t r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(p2(a)), "l"(p2(b)));
  return f2(r);
}
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) {
  uint64_t r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(p2(a)), "l"(p2(b)), "l"(p2(c)));
  return f2(r);
}
__device__ __forceinline__ float2 both(float v) { return make_float2(v, v); }
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return fma2(b, both(-1.0f), a); }
// 12 D of a pair across rows or planes: (m2 - p2) + 8 (p1 - m1)
__device__ __forceinline__ float2 c4p(float2 m2, float2 m1, float2 p1, float2 q2) {
  return fma2(both(8.0f), sub2(p1, m1), sub2(m2, q2));
}
// 12 D of the pair b along x, from the pairs before and after it
__device__ __forceinline__ float2 c4x(float2 a, float2 b, float2 e) {
  return fma2(both(8.0f), make_float2(b.y - a.y, e.x - b.x), sub2(a, e));
}

// Offset of node (x, y) of plane 0 in one padded component (32 bits: a
// component holds fewer than 2^31 nodes); plane z adds z * Geom::plane.
__device__ __forceinline__ int zm_off(const Geom& g, int x, int y) {
  return g.pz * (int)g.plane + (y + PAD) * g.np[0] + x + g.padx;
}

struct ZmOperands {  // update operands of one own node pair at one output plane
  float2 d[3], a[3], f[3], irh;
};

// Element access at a 32-bit byte offset from a base that is the same for the
// whole warp: one instruction, no 64-bit address arithmetic (a component is
// below 4 GB: plan_zmarch).
template <class V>
__device__ __forceinline__ V* zm_at(const float* base, unsigned bytes) {
  return reinterpret_cast<V*>(reinterpret_cast<char*>(const_cast<float*>(base)) + bytes);
}

// Update operands of the own pair at byte offset o of a component (full: both
// nodes are unknowns; else v0, v1); D, A, R: delta, acc and f/rho of this
// right-hand side, F the component stride.
template <int MODE, bool FORCED>
__device__ __forceinline__ void zm_load_ops(const float* D, const float* A, const float* R, const float* irh2,
                                            unsigned o, long long F, bool full, bool v0, bool v1, ZmOperands& op) {
  if (full) {  // 8-byte aligned: x - off[0] and the padded row start are even
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      if (MODE != STEP_FIRST) {
        op.d[c] = __ldcs(zm_at<const float2>(D + c * F, o));
        op.a[c] = __ldcs(zm_at<const float2>(A + c * F, o));
      }
      if (FORCED) op.f[c] = __ldg(zm_at<const float2>(R + c * F, o));
    }
    op.irh = __ldg(zm_at<const float2>(irh2, o));
  } else {
    auto ld = [&](const float* b) {
      return make_float2(v0 ? *zm_at<const float>(b, o) : 0.f, v1 ? *zm_at<const float>(b, o + 4) : 0.f);
    };
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      if (MODE != STEP_FIRST) op.d[c] = ld(D + c * F), op.a[c] = ld(A + c * F);
      if (FORCED) op.f[c] = ld(R + c * F);
    }
    op.irh = ld(irh2);
  }
}

// lambda, mu at the stress pair at byte offset o (zero outside the grid; full:
// both nodes lie in it, else g0, g1)
__device__ __forceinline__ void zm_load_lm(const float* lam, const float* mu, unsigned o, bool full, bool g0, bool g1,
                                           float2& l, float2& m) {
  if (full) {  // padded x even: 8-byte aligned
    l = __ldg(zm_at<const float2>(lam, o));
    m = __ldg(zm_at<const float2>(mu, o));
    return;
  }
  l = m = make_float2(0.f, 0.f);
  if (g0) l.x = __ldg(zm_at<const float>(lam, o)), m.x = __ldg(zm_at<const float>(mu, o));
  if (g1) l.y = __ldg(zm_at<const float>(lam, o + 4)), m.y = __ldg(zm_at<const float>(mu, o + 4));
}

// Leapfrog / filter update (increment form) of the own pair at byte offset p
// of a component from k = 144 h^2 rho M^{-1} K u; u of the pair at Us
// (component stride us).
template <int MODE, bool FORCED>
__device__ __forceinline__ void zm_update(const ZmScalars& sc, const ZmOperands& op, const float2 k[3], const float* Us,
                                          int us, float* D, float* A, float* U, unsigned p, long long F, bool full,
                                          bool v0, bool v1) {
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const float2 u = ld2(Us + c * us);
    float2 a = mul2(k[c], op.irh);
    if (FORCED) a = fma2(op.f[c], both(sc.fcos144), a);
    float2 d, ac;
    if (MODE == STEP_FIRST) d = mul2(both(-0.5f * sc.kt144), a);
    else d = fma2(both(-sc.kt144), a, op.d[c]);
    const float2 un = add2(u, d);
    if (MODE == STEP_FIRST) ac = fma2(both(sc.w0), u, mul2(both(sc.wnew), un));
    else ac = fma2(both(sc.wnew), un, op.a[c]);
    auto st = [&](float* b, float2 v) {
      if (full) {
        __stcs(zm_at<float2>(b, p), v);
      } else {
        if (v0) *zm_at<float>(b, p) = v.x;
        if (v1) *zm_at<float>(b, p + 4) = v.y;
      }
    };
    if (MODE != STEP_LAST) st(D + c * F, d), st(U + c * F, un);
    st(A + c * F, ac);
  }
}

// 12 D along x of the pair at v (8-byte aligned), class taps per node
__device__ __forceinline__ float2 zm_tap_pair_x(const float* v, int c0, int c1, const int* toff, const float* tcf) {
  return make_float2(zm_d12t(v, 1, c0, toff, tcf), zm_d12t(v + 1, 1, c1, toff, tcf));
}
__device__ __forceinline__ float2 zm_tap_pair_y(const float* v, int stride, int c, const int* toff, const float* tcf) {
  return make_float2(zm_d12t(v, stride, c, toff, tcf), zm_d12t(v + 1, stride, c, toff, tcf));
}

__device__ __forceinline__ bool zm_unknown_x(const Geom& g, int x) { return x >= g.off[0] && x < g.off[0] + g.nu[0]; }
__device__ __forceinline__ bool zm_unknown_y(const Geom& g, int y) { return y >= g.off[1] && y < g.off[1] + g.nu[1]; }

// A pair of stress nodes (x, x + 1) of row y: which lie in the grid, and the
// SBP classes along x and y.
struct ZmPair {
  bool g0, g1;
  int c0, c1, cy;
  __device__ __forceinline__ ZmPair(const Geom& g, int x, int y) {
    const bool in = y >= 0 && y < g.n[1];
    g0 = in && x >= 0 && x < g.n[0];
    g1 = in && x + 1 >= 0 && x + 1 < g.n[0];
    c0 = zm_class(x, g.n[0]);
    c1 = zm_class(x + 1, g.n[0]);
    cy = zm_class(y, g.n[1]);
  }
};

// 12 sigma at a pair of plane s (u ring at sm, pair at offset uo of a plane)
// into the in-plane buffer at offset ps; returns (xz, yz, zz).  lambda = mu = 0
// outside the grid.
template <class L>
__device__ __forceinline__ void zm_stress(const float* sm, float* sip, int uo, int ps, int s, bool zin, int n2,
                                          const ZmPair& p, bool wx, bool wy, float2 l, float2 m, const int* toff,
                                          const float* tcf, float2 out_z[3]) {
  const float* const U0 = sm + (s & (ZM_RU - 1)) * L::USLOT + uo;
  float2 dx[3], dy[3], dz[3];
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const float* Uc = U0 + c * L::UPLANE;
    dx[c] = wx ? zm_tap_pair_x(Uc, p.c0, p.c1, toff, tcf) : c4x(ld2(Uc - 2), ld2(Uc), ld2(Uc + 2));
    dy[c] = wy ? zm_tap_pair_y(Uc, L::UX, p.cy, toff, tcf)
               : c4p(ld2(Uc - 2 * L::UX), ld2(Uc - L::UX), ld2(Uc + L::UX), ld2(Uc + 2 * L::UX));
  }
  if (zin) {  // uniform per plane
    const float* const M2 = sm + ((s - 2) & (ZM_RU - 1)) * L::USLOT + uo;
    const float* const M1 = sm + ((s - 1) & (ZM_RU - 1)) * L::USLOT + uo;
    const float* const P1 = sm + ((s + 1) & (ZM_RU - 1)) * L::USLOT + uo;
    const float* const P2 = sm + ((s + 2) & (ZM_RU - 1)) * L::USLOT + uo;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const int o = c * L::UPLANE;
      dz[c] = c4p(ld2(M2 + o), ld2(M1 + o), ld2(P1 + o), ld2(P2 + o));
    }
  } else {
    const int cz = zm_class(s, n2);
#pragma unroll
    for (int c = 0; c < 3; ++c) dz[c] = make_float2(0.f, 0.f);
    for (int q = 0; q < 4; ++q) {
      const float* const P = sm + ((s + toff[4 * cz + q]) & (ZM_RU - 1)) * L::USLOT + uo;
      const float2 wq = both(tcf[4 * cz + q]);
#pragma unroll
      for (int c = 0; c < 3; ++c) dz[c] = fma2(wq, ld2(P + c * L::UPLANE), dz[c]);
    }
  }
  const float2 ld = mul2(l, add2(add2(dx[0], dy[1]), dz[2])), m2 = add2(m, m);
  const float2 sxx = fma2(m2, dx[0], ld), syy = fma2(m2, dy[1], ld), sxy = mul2(m, add2(dy[0], dx[1]));
  out_z[0] = mul2(m, add2(dz[0], dx[2]));
  out_z[1] = mul2(m, add2(dz[1], dy[2]));
  out_z[2] = fma2(m2, dz[2], ld);
  float* const S = sip + ps;
  st2(S, sxx.x, sxx.y);
  st2(S + L::SPLANE, syy.x, syy.y);
  st2(S + 2 * L::SPLANE, sxy.x, sxy.y);
  st2(S + 3 * L::SPLANE, out_z[0].x, out_z[0].y);
  st2(S + 4 * L::SPLANE, out_z[1].x, out_z[1].y);
}

template <int TX, int TY>
constexpr int zm_ctas() { return TX * TY <= 256 ? 2 : 1; }

template <int TX, int TY, int MODE, bool FORCED>
__global__ void __launch_bounds__(ZmLayout<TX, TY>::NT, zm_ctas<TX, TY>())
    step3d_o4_zm(Geom g, WaveFields<float> f, ZmScalars sc, unsigned* ctl, const __grid_constant__ CUtensorMap tmu) {
  using L = ZmLayout<TX, TY>;
  extern __shared__ unsigned char zm_raw[];
  // 128-byte aligned base; offsetting the shared array itself (rather than an
  // integer round trip) keeps every access below in the shared address space
  float* const sm = reinterpret_cast<float*>(zm_raw + ((128u - (smem_u32(zm_raw) & 127u)) & 127u));
  uint64_t* const bar = reinterpret_cast<uint64_t*>(sm + L::FLOATS);
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  int* const toff = reinterpret_cast<int*>(sm + L::OFF_CLS);
  float* const tcf = sm + L::OFF_CLS + 4 * ZM_CLASSES;
  if (t == 0) {  // static indices: the parameter arrays stay in the constant bank
#pragma unroll
    for (int k = 0; k < 4 * ZM_CLASSES; ++k) toff[k] = sc.toff[k], tcf[k] = sc.tcf[k];
    for (int k = 0; k < ZM_RU; ++k) mbar_init(bar + k, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  // this thread's stress pair: nodes (X0 + 2 pi, + 1), row Y0 + ri
  const bool own = warp < L::NWO;
  int pi = lane % L::PW, ri;
  if (own) {
    ri = warp * L::RPW + lane / L::PW;
  } else {
    const int k = (warp - L::NWO) * L::RPW + lane / L::PW;  // rows -2, -1, TY, TY + 1
    ri = k < 2 ? k - 2 : TY + k - 2;
  }
  const int uo = (ri + 4) * L::UX + 4 + 2 * pi;  // of the pair in a u plane
  const int ps = (ri + 2) * L::SX + 2 + 2 * pi;  // ... in a stress plane
  // the first halo warp takes the left and right halo pairs of the own rows in a second pass
  const bool two = warp == L::NWO, xside = two && lane < 2 * TY;
  const int xpi = (lane & 1) ? L::PW : -1, xri = lane >> 1;
  __syncthreads();
  zm_pdl_wait();
  zm_pdl_trigger();
  const unsigned long long wait_ns = *reinterpret_cast<const volatile unsigned long long*>(ctl + 2);

  const int n0 = g.n[0], n1 = g.n[1], n2 = g.n[2];
  const int ntx = (g.nu[0] + sc.shx + TX - 1) / TX, nty = (g.nu[1] + sc.shy + TY - 1) / TY, nz = g.nu[2];
  const long long W = (long long)ntx * nty * nz * g.nrhs;
  const long long wbeg = W * blockIdx.x / gridDim.x, wend = W * (blockIdx.x + 1) / gridDim.x;
  const long long F = g.field;
  const unsigned PL4 = 4u * (unsigned)g.plane;  // bytes of a plane
  const float BT = sc.bt12;
  unsigned phase = 0;  // parity of the next completion of each u slot's mbarrier
  bool alive = true;
  long long w = wbeg;

  while (w < wend && alive) {
    // ---- segment: tile (rhs, tx, ty), output planes [za, zb)
    const long long tile = w / nz;
    const int zi = (int)(w - tile * nz);
    const int zcount = (int)((wend - w) < (long long)(nz - zi) ? (wend - w) : (long long)(nz - zi));
    w += zcount;
    const int rhs = (int)(tile / (ntx * nty));
    const int tt = (int)(tile - (long long)rhs * ntx * nty);
    const int X0 = g.off[0] - sc.shx + TX * (tt % ntx), Y0 = g.off[1] - sc.shy + TY * (tt / ntx);
    const int za = g.off[2] + zi, zb = za + zcount;
    // stress planes [slo, shi] the outputs read; u planes [ulo, uhi] those read
    const int slo = min(zm_lo(za, n2), zm_lo(zb - 1, n2)), shi = max(zm_hi(za, n2), zm_hi(zb - 1, n2));
    const int ulo = min(zm_lo(slo, n2), zm_lo(shi, n2)), uhi = max(zm_hi(slo, n2), zm_hi(shi, n2));
    // bulk-tensor coordinates of the u box (padded x is a multiple of 4: Geom::padx)
    const int cx = X0 - 4 + g.padx, cy = Y0 - 4 + PAD, cc = 3 * rhs;
    int issued = min(uhi, slo + 3);  // last u plane requested
    __syncthreads();  // every read of the rings by the previous segment is done
    if (t == 0) {
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      for (int k = ulo; k <= issued; ++k)
        zm_issue(&tmu, sm + (k & (ZM_RU - 1)) * L::USLOT, bar + (k & (ZM_RU - 1)), cx, cy, k + g.pz, cc,
                 L::TX_BYTES);
    }
    const int sx = X0 + 2 * pi, sy = Y0 + ri;
    const bool ov0 = own && zm_unknown_x(g, sx) && zm_unknown_y(g, sy);
    const bool ov1 = own && zm_unknown_x(g, sx + 1) && zm_unknown_y(g, sy);
    const bool live = ov0 || ov1;
    const ZmPair pm(g, sx, sy);
    // warps with a lane on an SBP closure row take that axis by the class taps
    const bool wx = __any_sync(0xffffffffu, pm.c0 != 4 || pm.c1 != 4), wy = __any_sync(0xffffffffu, pm.cy != 4);
    const unsigned so = 4u * (unsigned)zm_off(g, sx, sy);  // byte offset of this thread's pair at plane 0
    const bool fs = pm.g0 && pm.g1, fo = ov0 && ov1;
    const long long ro = (long long)rhs * 3 * g.field;
    float* const Dr = f.delta + ro;
    float* const Ar = f.acc + ro;
    float* const Ur = f.u_next + ro;
    const float* const Rr = FORCED ? f.frho + ro : nullptr;
    // own column of the closure planes near the z sides: z stresses (0..2) and
    // in-plane sums (3..5), written and read by this thread only
    float* const Sg = f.sigma + (long long)rhs * 6 * g.field;
    float2 lm_l, lm_m;  // lambda, mu of the next stress plane, requested one plane ahead
    zm_load_lm(f.lam, f.mu, so + slo * PL4, fs, pm.g0, pm.g1, lm_l, lm_m);
    // 144 h^2 rho M^{-1} K u of the outputs s - 2 .. s + 1 as far as planes < s give it
    float2 A0[3], A1[3], A2[3], A3[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) A0[c] = A1[c] = A2[c] = A3[c] = make_float2(0.f, 0.f);

    int have = ulo - 1, next_o = za;  // last u plane waited for, next output
    int s = slo;
    for (; s <= shi; ++s) {
      // ---- wait for the u planes that stress plane s reads (bounded)
      bool bad = false;
      const int need = max(have, zm_hi(s, n2));
      for (int k = have + 1; k <= need && !bad; ++k) {
        const int sl = k & (ZM_RU - 1);
        const unsigned par = (phase >> sl) & 1u;
        bool ok = wait_ns != 0ull;
        if (ok && !mbar_try(bar + sl, par)) {
          const unsigned long long t0 = zm_ns();
          while (!mbar_try(bar + sl, par)) {
            if (zm_ns() - t0 > wait_ns) {
              ok = false;
              break;
            }
          }
        }
        if (ok) phase ^= 1u << sl, have = k;
        bad = !ok;
      }
      // ---- 12 sigma at the pair (and at the side pair of the first halo warp)
      float* const sip = sm + L::OFF_SIP + (s & 1) * L::SBUF;
      const bool zin = s >= 4 && s <= n2 - 5;
      float2 own_z[3];
      zm_stress<L>(sm, sip, uo, ps, s, zin, n2, pm, wx, wy, lm_l, lm_m, toff, tcf, own_z);
      if (two) {
        const ZmPair px(g, X0 + 2 * xpi, Y0 + xri);
        const bool vx = xside && (px.c0 != 4 || px.c1 != 4), vy = xside && px.cy != 4;
        const bool xx = __any_sync(0xffffffffu, vx), xy = __any_sync(0xffffffffu, vy);
        if (xside) {
          float2 xl, xm, unused[3];
          zm_load_lm(f.lam, f.mu, 4u * (unsigned)zm_off(g, X0 + 2 * xpi, Y0 + xri) + s * PL4, px.g0 && px.g1, px.g0, px.g1,
                     xl, xm);
          zm_stress<L>(sm, sip, (xri + 4) * L::UX + 4 + 2 * xpi, (xri + 2) * L::SX + 2 + 2 * xpi, s, zin, n2, px, xx, xy,
                       xl, xm, toff, tcf, unused);
        }
      }
      // operands of the next stress plane and of this step's output, in flight across the barrier
      if (s + 1 <= shi) zm_load_lm(f.lam, f.mu, so + (s + 1) * PL4, fs, pm.g0, pm.g1, lm_l, lm_m);
      const int o = s - 2;
      const bool out = o >= max(za, 4) && o <= min(zb - 1, n2 - 5);
      ZmOperands op;
      if (out && live) zm_load_ops<MODE, FORCED>(Dr, Ar, Rr, f.irh2, so + o * PL4, F, fo, ov0, ov1, op);
      // the stress plane is complete (or a wait gave up: every thread stops);
      // every read of planes below s - 3 and of the other stress buffer is done
      if (__syncthreads_or(bad)) {
        alive = false;
        break;
      }
      if (t == 0 && s + 4 <= uhi && s + 4 > issued) {
        const int k = (s + 4) & (ZM_RU - 1);
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        zm_issue(&tmu, sm + k * L::USLOT, bar + k, cx, cy, s + 4 + g.pz, cc, L::TX_BYTES);
      }
      issued = max(issued, min(uhi, s + 4));
      if (live) {
        // in-plane part of -D sigma + H^{-1} B sigma at plane s
        constexpr int CX[3] = {0, 2, 3}, CY[3] = {2, 1, 4};  // planes of sigma_{cx}, sigma_{cy}
        float2 kp[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          const float* Sx = sip + CX[c] * L::SPLANE + ps;
          const float* Sy = sip + CY[c] * L::SPLANE + ps;
          const float2 kx = wx ? zm_tap_pair_x(Sx, pm.c0, pm.c1, toff, tcf) : c4x(ld2(Sx - 2), ld2(Sx), ld2(Sx + 2));
          const float2 ky = wy ? zm_tap_pair_y(Sy, L::SX, pm.cy, toff, tcf)
                               : c4p(ld2(Sy - 2 * L::SX), ld2(Sy - L::SX), ld2(Sy + L::SX), ld2(Sy + 2 * L::SX));
          kp[c] = make_float2(-(kx.x + ky.x), -(kx.y + ky.y));
          if (wx || wy) {  // boundary terms H^{-1} B sigma on free sides (nodes on the side itself)
            float b0 = 0.f, b1 = 0.f;
            if (sx == 0) b0 -= BT * Sx[0];
            if (sx == n0 - 1) b0 += BT * Sx[0];
            if (sx + 1 == n0 - 1) b1 += BT * Sx[1];
            if (sy == 0) b0 -= BT * Sy[0], b1 -= BT * Sy[1];
            if (sy == n1 - 1) b0 += BT * Sy[0], b1 += BT * Sy[1];
            kp[c].x += b0;
            kp[c].y += b1;
          }
        }
        // plane s enters the outputs s - 2 .. s + 2
        float2 k[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          const float2 z = own_z[c];
          k[c] = add2(A0[c], z);
          A0[c] = fma2(both(-8.0f), z, A1[c]);
          A1[c] = add2(A2[c], kp[c]);
          A2[c] = fma2(both(8.0f), z, A3[c]);
          A3[c] = make_float2(-z.x, -z.y);
        }
        const bool near = s <= 5 || s >= n2 - 6;
        if (near) {  // the outputs on z closure rows read these planes back
#pragma unroll
          for (int c = 0; c < 3; ++c) {
            *zm_at<float2>(Sg + c * F, so + s * PL4) = own_z[c];
            *zm_at<float2>(Sg + (3 + c) * F, so + s * PL4) = kp[c];
          }
        }
        if (out)
          zm_update<MODE, FORCED>(sc, op, k, sm + (o & (ZM_RU - 1)) * L::USLOT + uo, L::UPLANE, Dr, Ar, Ur, so + o * PL4,
                                  F, fo, ov0, ov1);
      }
      if (out) next_o = o + 1;
      // ---- outputs on z closure rows whose stress planes all exist
      for (; next_o < zb && (next_o < 4 || next_o > n2 - 5) && zm_hi(next_o, n2) <= s; ++next_o) {
        if (!live) continue;
        const int oz = next_o, cz = zm_class(oz, n2);
        const unsigned q = so + oz * PL4;
        ZmOperands po;
        zm_load_ops<MODE, FORCED>(Dr, Ar, Rr, f.irh2, q, F, fo, ov0, ov1, po);
        float2 k[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
          k[c] = *zm_at<float2>(Sg + (3 + c) * F, q);
          for (int j = 0; j < 4; ++j)
            k[c] = fma2(both(-tcf[4 * cz + j]), *zm_at<float2>(Sg + c * F, q + toff[4 * cz + j] * PL4), k[c]);
          if (oz == 0 || oz == n2 - 1) k[c] = fma2(both(oz == 0 ? -BT : BT), *zm_at<float2>(Sg + c * F, q), k[c]);
        }
        zm_update<MODE, FORCED>(sc, po, k, sm + (oz & (ZM_RU - 1)) * L::USLOT + uo, L::UPLANE, Dr, Ar, Ur, q, F, fo,
                                ov0, ov1);
      }
    }
    if (!alive) {
      // wait (bounded) for this segment's copies still in flight, then stop
      if (t == 0) atomicAdd(ctl + 4, 1u);
      const unsigned long long t0 = zm_ns();
      for (int k = have + 1; k <= issued; ++k) {  // requested, not yet consumed
        const int sl = k & (ZM_RU - 1);
        while (!mbar_try(bar + sl, (phase >> sl) & 1u) && zm_ns() - t0 < 1000000000ull) {
        }
        phase ^= 1u << sl;
      }
      // the accumulator of every remaining own output is NaN
      const float nanv = __int_as_float(0x7fc00000);
      for (long long ww = w - zcount + (next_o - za); own && ww < wend;) {
        const long long tl = ww / nz;
        const int z0 = (int)(ww - tl * nz);
        const int cnt = (int)((wend - ww) < (long long)(nz - z0) ? (wend - ww) : (long long)(nz - z0));
        const int rh = (int)(tl / (ntx * nty));
        const int t2 = (int)(tl - (long long)rh * ntx * nty);
        const int x = g.off[0] - sc.shx + TX * (t2 % ntx) + 2 * pi, y = g.off[1] - sc.shy + TY * (t2 / ntx) + ri;
        for (int zz = 0; zz < cnt; ++zz)
          for (int e = 0; e < 2; ++e)
            if (zm_unknown_x(g, x + e) && zm_unknown_y(g, y))
              for (int c = 0; c < 3; ++c) f.acc[pidx(g, rh, c, x + e, y, g.off[2] + z0 + zz)] = nanv;
        ww += cnt;
      }
    }
  }
}

// ---- host side ----------------------------------------------------------------
template <int TX, int TY>
cudaError_t zm_map(const Geom& g, const float* u, unsigned char* out) {
  static_assert(sizeof(CUtensorMap) <= ZM_MAP_BYTES, "tensor map storage");
  EncodeTiledFn enc = encode_fn();
  if (!enc) return cudaErrorNotSupported;
  const cuuint64_t dims[4] = {(cuuint64_t)g.np[0], (cuuint64_t)g.np[1], (cuuint64_t)g.np[2],
                              (cuuint64_t)(3 * g.nrhs)};
  const cuuint64_t strides[3] = {(cuuint64_t)g.np[0] * sizeof(float), (cuuint64_t)g.plane * sizeof(float),
                                 (cuuint64_t)g.field * sizeof(float)};
  const cuuint32_t box[4] = {(cuuint32_t)(TX + 8), (cuuint32_t)(TY + 8), 1, 3};
  const cuuint32_t es[4] = {1, 1, 1, 1};
  CUtensorMap m;
  const CUresult rc = enc(&m, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 4, const_cast<float*>(u), dims, strides, box, es,
                          CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_128B,
                          CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (rc != CUDA_SUCCESS) return cudaErrorInvalidValue;
  std::memcpy(out, &m, sizeof(m));
  return cudaSuccess;
}

template <int TX, int TY>
void* zm_kernel(int mode, bool forced) {
  if (mode == STEP_FIRST)
    return forced ? (void*)step3d_o4_zm<TX, TY, STEP_FIRST, true> : (void*)step3d_o4_zm<TX, TY, STEP_FIRST, false>;
  if (mode == STEP_MID)
    return forced ? (void*)step3d_o4_zm<TX, TY, STEP_MID, true> : (void*)step3d_o4_zm<TX, TY, STEP_MID, false>;
  return forced ? (void*)step3d_o4_zm<TX, TY, STEP_LAST, true> : (void*)step3d_o4_zm<TX, TY, STEP_LAST, false>;
}


template <int TX, int TY>
void plan_one(const Geom& g, const float* u_a, const float* u_b, int sms, int smem_max, ZmPlan& p, int k) {
  using L = ZmLayout<TX, TY>;
  p.ok[k] = 0;
  // x: a multiple of 4 keeps the bulk-tensor box 16-byte aligned and the node pairs even
  p.shx[k] = zm_shift(g.nu[0], TX, g.hi_free[0] != 0, 4);
  p.shy[k] = zm_shift(g.nu[1], TY, g.hi_free[1] != 0, 1);
  if (p.shx[k] < 0 || p.shy[k] < 0 || (int)L::BYTES > smem_max) return;
  for (int mode = 0; mode < 3; ++mode)
    for (int fo = 0; fo < 2; ++fo)
      if (cudaFuncSetAttribute(zm_kernel<TX, TY>(mode, fo != 0), cudaFuncAttributeMaxDynamicSharedMemorySize,
                               (int)L::BYTES) != cudaSuccess) {
        cudaGetLastError();
        return;
      }
  int per_sm = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, zm_kernel<TX, TY>(STEP_MID, false), L::NT, L::BYTES) !=
          cudaSuccess ||
      per_sm < 1) {
    cudaGetLastError();
    return;
  }
  if (zm_map<TX, TY>(g, u_a, p.tmap[k][0]) != cudaSuccess || zm_map<TX, TY>(g, u_b, p.tmap[k][1]) != cudaSuccess) {
    cudaGetLastError();
    return;
  }
  const long long tiles =
      (long long)((g.nu[0] + p.shx[k] + TX - 1) / TX) * ((g.nu[1] + p.shy[k] + TY - 1) / TY) * g.nrhs;
  const long long work = tiles * g.nu[2];
  long long grid = (long long)per_sm * sms;
  const char* cap = getenv("EWH_ZM_GRID");  // fewer CTAs: longer (tile, z range) shares per CTA
  if (cap && atoi(cap) > 0 && atoi(cap) < grid) grid = atoi(cap);
  if (grid > work) grid = work;
  p.grid[k] = (int)grid;
  p.ok[k] = 1;
  if (getenv("EWH_VERBOSE"))
    fprintf(stderr,
            "ewh: z-march plan %d (%d x %d): %lld tiles (shift %d, %d) x %d planes on %lld CTAs (%d per SM), %zu B "
            "shared\n",
            k, TX, TY, tiles, p.shx[k], p.shy[k], g.nu[2], grid, per_sm, (size_t)L::BYTES);
}

template <int TX, int TY, int MODE>
cudaError_t zm_launch(const cudaLaunchConfig_t& cfg, bool forced, const Geom& g, const WaveFields<float>& f,
                      const ZmScalars& sc, unsigned* ctl, const CUtensorMap& tm) {
  return forced ? cudaLaunchKernelEx(&cfg, step3d_o4_zm<TX, TY, MODE, true>, g, f, sc, ctl, tm)
                : cudaLaunchKernelEx(&cfg, step3d_o4_zm<TX, TY, MODE, false>, g, f, sc, ctl, tm);
}

template <int TX, int TY>
cudaError_t zm_launch_mode(cudaLaunchConfig_t& cfg, StepMode mode, bool forced, const Geom& g,
                           const WaveFields<float>& f, const ZmScalars& sc, unsigned* ctl, const CUtensorMap& tm) {
  cfg.blockDim = dim3(ZmLayout<TX, TY>::NT);
  cfg.dynamicSmemBytes = ZmLayout<TX, TY>::BYTES;
  if (mode == STEP_FIRST) return zm_launch<TX, TY, STEP_FIRST>(cfg, forced, g, f, sc, ctl, tm);
  if (mode == STEP_MID) return zm_launch<TX, TY, STEP_MID>(cfg, forced, g, f, sc, ctl, tm);
  return zm_launch<TX, TY, STEP_LAST>(cfg, forced, g, f, sc, ctl, tm);
}

}  // namespace

// Build the fused-kernel plan of a 3D order-4 FP32 context: tensor maps of
// both u buffers per shape, the persistent grids, the shared-memory opt-in.
// A shape is unusable (the per-level pair runs) when the geometry is outside
// what the kernel handles: fewer than 12 planes along z, or 4 GB and more per
// component (32-bit byte offsets).
ZmPlan plan_zmarch(const Geom& g, const float* u_a, const float* u_b, unsigned* ctl) {
  ZmPlan p;
  if (g.dim != 3 || g.mapped || g.n[2] < 12 || g.off[0] + g.padx != 8 || g.field >= (1LL << 30)) return p;
  int dev = 0, sms = 0, smem_max = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&smem_max, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev) != cudaSuccess) {
    cudaGetLastError();
    return p;
  }
  plan_one<64, 8>(g, u_a, u_b, sms, smem_max, p, 0);
  plan_one<32, 8>(g, u_a, u_b, sms, smem_max, p, 1);
  p.u_a = u_a;
  p.u_b = u_b;
  p.ctl = ctl;
  return p;
}

cudaError_t launch_zmarch(const Geom& g, const ZmPlan& p, int k, const WaveFields<float>& f, StepMode mode,
                          const StepScalars& s, cudaStream_t st) {
  if (k < 0 || k >= ZM_SHAPES || !p.ok[k]) return cudaErrorInvalidValue;
  const int b = f.u_cur == p.u_a ? 0 : (f.u_cur == p.u_b ? 1 : -1);
  if (b < 0) return cudaErrorInvalidValue;
  CUtensorMap tm;
  std::memcpy(&tm, p.tmap[k][b], sizeof(tm));
  ZmScalars sc;
  sc.kt144 = (float)(s.kt / 144.0);
  sc.w0 = (float)s.w0;
  sc.wnew = (float)s.wnew;
  sc.fcos144 = (float)(144.0 * s.cosn);
  sc.bt12 = (float)(12.0 * 48.0 / 17.0);
  sc.shx = p.shx[k];
  sc.shy = p.shy[k];
  zm_class_taps(sc.toff, sc.tcf);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(p.grid[k]);
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  const char* e = getenv("EWH_PDL");
  cfg.numAttrs = (e && e[0] == '0') ? 0 : 1;
  const bool forced = f.frho != nullptr;
  return k == 0 ? zm_launch_mode<64, 8>(cfg, mode, forced, g, f, sc, p.ctl, tm)
                : zm_launch_mode<32, 8>(cfg, mode, forced, g, f, sc, p.ctl, tm);
}

}  // namespace ewh
