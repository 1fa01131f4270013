// Order 4 (SBP), 2D, FP64: one fused launch per leapfrog level in block fixed
// point (ewh_fixed.cuh).  It computes the level of the time-corrected explicit
// scheme (Section 4.3, eq. elastic-time-explicit-corrected) in increment form
// with the trapezoid accumulation of eq. (qoper).
//
// A CTA owns 32 x TY nodes.  It
//   - loads u^n on the tile +- 4 nodes and lambda, mu on the tile +- 2, and
//     takes the largest exponent of each over the tile;
//   - quantises u to integers up to 2^57 in shared memory;
//   - forms 12 sigma on the tile +- 2 (exact differences, upper halves of the
//     products with lambda and 2 mu);
//   - differences them exactly, converts the sum to FP64 and applies the
//     leapfrog / filter update in FP64, as the other kernels do.
// Every intermediate stays below 2^63 for any input: the weights of 12 D add up
// to 18 in the interior and at most 41.6 on a closure row, so tiles with closure
// rows scale lambda and mu down by one more bit and add their parts in FP64.
//
// Per node that leaves 9 FP64 instructions of 42; the rest are integer ones.  At
// 1026 x 1026 nodes a level takes 42 us, against 105 us for the FP64 stress +
// divergence pair, whose FP64 pipe is full (now 43%, integer 41%, issue 54%).
// Error of S v against 80-bit arithmetic (layered, random and mixed media, 220 to
// 300 nodes a side; waves, noise, point sources): 0.7 .. 3.0e-15, the pair 0.7 ..
// 3.4e-15.  Tiles of 16 and 8 rows: the smaller ones fill the GPU on small grids
// (the autotuner picks).  A tile that holds an infinity or a NaN, magnitudes next to the largest
// FP64 numbers, or a medium whose moduli differ by more than 2^FX_CONTRAST
// (a stress keeps its bits below the tile's stiffest node) takes a plain FP64
// path.
#include <cuda_runtime.h>
#include <stdint.h>

#include <cstdlib>

#include "ewh_fixed.cuh"
#include "ewh_internal.cuh"
#include "ewh_march.cuh"

namespace ewh {
namespace {

// 12 sigma at a grid node in FP64 from global u (the plain path)
__device__ void fx_sigma_plain(const double* U, long long fld, int sy, double l, double m, int cx, int cy,
                               const FxTaps& tp, double s[3]) {
  double ux = 0.0, uy = 0.0, vx = 0.0, vy = 0.0;
  for (int q = 0; q < 4; ++q) {
    const double wx = (double)tp.w[4 * cx + q] * fx_pow2(-FX_TAP), wy = (double)tp.w[4 * cy + q] * fx_pow2(-FX_TAP);
    const int ox = tp.off[4 * cx + q], oy = tp.off[4 * cy + q] * sy;
    if (wx != 0.0) ux += wx * U[ox], vx += wx * U[ox + fld];
    if (wy != 0.0) uy += wy * U[oy], vy += wy * U[oy + fld];
  }
  s[0] = l * (ux + vy) + 2.0 * m * ux;
  s[1] = l * (ux + vy) + 2.0 * m * vy;
  s[2] = m * (uy + vx);
}

// 144 h^2 rho M^{-1} K u at node (x, y) in FP64
__device__ __noinline__ void fx_accel_plain(const Geom& g, const double* u, const double* lam, const double* mu,
                                            int rhs, int x, int y, const FxTaps& tp, double& ku, double& kv) {
  const int sy = g.np[0], cx = zm_class(x, g.n[0]), cy = zm_class(y, g.n[1]);
  const double* U = u + pidx(g, rhs, 0, x, y, 0);
  const long long pc = pidx(g, 0, 0, x, y, 0);
  const double bt = 12.0 * 48.0 / 17.0;
  double s[3];
  ku = kv = 0.0;
  for (int q = 0; q < 4; ++q) {
    const double wx = (double)tp.w[4 * cx + q] * fx_pow2(-FX_TAP), wy = (double)tp.w[4 * cy + q] * fx_pow2(-FX_TAP);
    if (wx != 0.0) {
      const int o = tp.off[4 * cx + q];
      fx_sigma_plain(U + o, g.field, sy, lam[pc + o], mu[pc + o], zm_class(x + o, g.n[0]), cy, tp, s);
      ku -= wx * s[0];
      kv -= wx * s[2];
    }
    if (wy != 0.0) {
      const int o = tp.off[4 * cy + q];
      fx_sigma_plain(U + o * sy, g.field, sy, lam[pc + o * sy], mu[pc + o * sy], cx, zm_class(y + o, g.n[1]), tp, s);
      ku -= wy * s[2];
      kv -= wy * s[1];
    }
  }
  const bool xe = x == 0 || x == g.n[0] - 1, ye = y == 0 || y == g.n[1] - 1;
  if (xe || ye) {
    fx_sigma_plain(U, g.field, sy, lam[pc], mu[pc], cx, cy, tp, s);
    if (xe) ku += x == 0 ? -bt * s[0] : bt * s[0], kv += x == 0 ? -bt * s[2] : bt * s[2];
    if (ye) ku += y == 0 ? -bt * s[2] : bt * s[2], kv += y == 0 ? -bt * s[1] : bt * s[1];
  }
}

constexpr int FX_TX = 32;                        // own columns of a tile: one warp per row
constexpr int FX_UX = FX_TX + 8, FX_SX = FX_TX + 4;  // u and stress tile rows

template <int TY>
struct Fx2 {
  static constexpr int NT = 16 * TY;                      // two own rows per warp
  static constexpr int UY = TY + 8, SY = TY + 4;
  static constexpr int UN = FX_UX * UY, SN = FX_SX * SY;  // positions of a tile
  static constexpr int OFF_S = 2 * UN;                    // in 64-bit words
  static constexpr int OFF_W = OFF_S + 3 * SN;            // tap weights, then offsets (ints), then keys
  static constexpr int OFF_O = OFF_W + 36;
  static constexpr int OFF_K = OFF_O + 18;
  static constexpr size_t BYTES = 8 * (size_t)(OFF_K + 32);
};

struct FxStep {
  double kt, kt144;  // c dt^2, c dt^2 / 144
  double fc;         // c dt^2 cos(w t_n)
  double w0, wnew;
  int shx, shy;      // tile origins: off - sh + tile size x index (zm_shift)
  i64 bt;            // 12 * 48 / 17 scaled by 2^FX_TAP
};

// Leapfrog / filter update of one value: k cs = -c dt^2 M^{-1} K u, fr = f / rho.
template <int MODE, bool FORCED>
__device__ __forceinline__ void fx_update(const WaveFields<double>& f, long long p, double u, double dp, double ap,
                                          double k, double cs, const FxStep& s) {
  const double fr = FORCED ? __ldg(f.frho + p) : 0.0;
  if (MODE == STEP_FIRST) {
    double d = k * cs;
    if (FORCED) d = fma(-s.fc, fr, d);
    d *= 0.5;
    const double un = u + d;
    f.delta[p] = d;
    f.u_next[p] = un;
    f.acc[p] = s.w0 * u + s.wnew * un;
  } else {
    double d = fma(k, cs, dp);
    if (FORCED) d = fma(-s.fc, fr, d);
    const double un = u + d;
    if (MODE == STEP_MID) {
      f.delta[p] = d;
      f.u_next[p] = un;
    }
    f.acc[p] = fma(s.wnew, un, ap);
  }
}

// Position k of thread (warp, lane) in a tile of W x H positions: the first 32
// columns row by row (row = warp + k NW), then the W - 32 others, several rows
// a warp.  Returns false when there is none.
template <int W, int H, int NW>
__device__ __forceinline__ bool fx_pos(int k, int warp, int lane, int& qx, int& qy) {
  constexpr int R = W - 32, PER = 32 / R;  // PER rows of the rest per warp
  qy = warp + k * NW;
  qx = lane;
  if (qy < H) return true;
  const int i = qy - H;  // the rest: PER rows each
  qx = 32 + lane % R;
  qy = i * PER + lane / R;
  return qy < H;
}

template <int MODE, bool FORCED, int TY, int MINB>
__global__ void __launch_bounds__(Fx2<TY>::NT, MINB)
    step2d_o4_fx(Geom g, WaveFields<double> f, FxStep s, const __grid_constant__ FxTaps tp) {
  using L = Fx2<TY>;
  constexpr int NW = L::NT / 32;
  constexpr int KU = (L::UY + (L::UY + 3) / 4 + NW - 1) / NW;  // 8 more columns: 4 rows a warp
  constexpr int KS = (L::SY + (L::SY + 7) / 8 + NW - 1) / NW;  // 4 more columns: 8 rows a warp
  static_assert(KU * NW >= L::UY + (L::UY + 3) / 4 && KS * NW >= L::SY + (L::SY + 7) / 8, "every position has a thread");
  extern __shared__ i64 fx_smem[];
  i64* const qu = fx_smem;
  i64* const sg = fx_smem + L::OFF_S;
  i64* const tw = fx_smem + L::OFF_W;
  int* const to = reinterpret_cast<int*>(fx_smem + L::OFF_O);
  unsigned* const keys = reinterpret_cast<unsigned*>(fx_smem + L::OFF_K);
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const int n0 = g.n[0], n1 = g.n[1], rhs = blockIdx.z;
  const int X0 = g.off[0] - s.shx + FX_TX * (int)blockIdx.x, Y0 = g.off[1] - s.shy + TY * (int)blockIdx.y;
  const int F = (int)g.field, npx = g.np[0];
  const int o0 = (Y0 + PAD) * npx + X0 + g.padx;  // padded offset of tile node (0, 0) in a component
  if (t < 36) tw[t] = tp.w[t], to[t] = tp.off[t];
  // lambda, mu of this thread's stress positions (static: ahead of the previous level's end)
  double l[KS], m[KS];
  unsigned km = 0, kn = 0x7fffffffu;  // largest of |lambda|, mu; smallest mu
#pragma unroll
  for (int k = 0; k < KS; ++k) {
    int qx, qy;
    const bool has = fx_pos<FX_SX, L::SY, NW>(k, warp, lane, qx, qy);
    const bool in = has && (unsigned)(X0 - 2 + qx) < (unsigned)n0 && (unsigned)(Y0 - 2 + qy) < (unsigned)n1;
    const int o = o0 + (qy - 2) * npx + qx - 2;
    l[k] = in ? __ldg(f.lam + o) : 0.0;
    m[k] = in ? __ldg(f.mu + o) : 0.0;
    km = max(km, max(fx_key(l[k]), fx_key(m[k])));
    if (in) kn = min(kn, fx_key(m[k]));
  }
  zm_pdl_wait();
  zm_pdl_trigger();
  const long long ro = (long long)rhs * 2 * g.field;
  const double* const U = f.u_cur + ro;
  double a[KU], b[KU];
  unsigned ku = 0;
#pragma unroll
  for (int k = 0; k < KU; ++k) {
    int qx, qy;
    const bool has = fx_pos<FX_UX, L::UY, NW>(k, warp, lane, qx, qy);
    const bool in = has && (unsigned)(X0 - 4 + qx) < (unsigned)n0 && (unsigned)(Y0 - 4 + qy) < (unsigned)n1;
    const int o = o0 + (qy - 4) * npx + qx - 4;
    a[k] = in ? U[o] : 0.0;
    b[k] = in ? U[o + F] : 0.0;
    ku = max(ku, max(fx_key(a[k]), fx_key(b[k])));
  }
  ku = __reduce_max_sync(0xffffffffu, ku);
  km = __reduce_max_sync(0xffffffffu, km);
  kn = __reduce_min_sync(0xffffffffu, kn);
  if (lane == 0) keys[3 * warp] = ku, keys[3 * warp + 1] = km, keys[3 * warp + 2] = kn;
  __syncthreads();
  ku = __reduce_max_sync(0xffffffffu, lane < NW ? keys[3 * lane] : 0u);
  km = __reduce_max_sync(0xffffffffu, lane < NW ? keys[3 * lane + 1] : 0u);
  kn = __reduce_min_sync(0xffffffffu, lane < NW ? keys[3 * lane + 2] : 0x7fffffffu);
  const bool edge = X0 - 2 < 4 || X0 + FX_TX + 1 > n0 - 5 || Y0 - 2 < 4 || Y0 + TY + 1 > n1 - 5;
  const int E = ku ? (int)(ku >> 20) : 1023, M0 = km ? (int)(km >> 20) : 1023;
  const int M = M0 + (edge ? 1 : 0);
  // u = q 2^(E-1022-57), lambda = q 2^(M-1022-58), the product's lower 64 bits dropped
  const int X = (E - 1022 - 57) + (M - 1022 - 58) + 64;
  if (ku >= 0x7ff00000u || M0 < 400 || M0 > 1600 || X > 950 || M0 - (int)(kn >> 20) > FX_CONTRAST) {  // plain FP64 (uniform per CTA)
#pragma unroll 1
    for (int k = 0; k < 2; ++k) {
      const int x = X0 + lane, y = Y0 + warp + k * NW;
      if (!is_unknown(g, x, y, 0)) continue;
      double au, av;
      fx_accel_plain(g, f.u_cur, f.lam, f.mu, rhs, x, y, tp, au, av);
      const double c = f.irh2[pidx(g, 0, 0, x, y, 0)] * s.kt144;
#pragma unroll 1
      for (int e = 0; e < 2; ++e) {
        const long long p = pidx(g, rhs, e, x, y, 0);
        const bool first = MODE == STEP_FIRST;
        fx_update<MODE, FORCED>(f, p, f.u_cur[p], first ? 0.0 : f.delta[p], first ? 0.0 : f.acc[p], e ? av : au, -c, s);
      }
    }
    return;
  }
#pragma unroll
  for (int k = 0; k < KU; ++k) {
    int qx, qy;
    if (fx_pos<FX_UX, L::UY, NW>(k, warp, lane, qx, qy)) {
      const int i = qy * FX_UX + qx;
      qu[i] = fx_from<57, true>(a[k], E);
      qu[L::UN + i] = fx_from<57, true>(b[k], E);
    }
  }
  // operands of the update, in flight during the stresses
  const int x = X0 + lane;
  const bool xu = x >= g.off[0] && x < g.off[0] + g.nu[0];
  double u0[2], u1[2], d0[2], d1[2], a0[2], a1[2], c[2];
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    const int y = Y0 + warp + k * NW;
    const bool un = xu && y >= g.off[1] && y < g.off[1] + g.nu[1];
    const int o = o0 + (warp + k * NW) * npx + lane;
    const long long p = ro + o;
    u0[k] = un ? U[o] : 0.0;
    u1[k] = un ? U[o + F] : 0.0;
    c[k] = un ? __ldg(f.irh2 + o) : 0.0;
    if (MODE != STEP_FIRST) {
      d0[k] = un ? f.delta[p] : 0.0, d1[k] = un ? f.delta[p + F] : 0.0;
      a0[k] = un ? f.acc[p] : 0.0, a1[k] = un ? f.acc[p + F] : 0.0;
    }
  }
  __syncthreads();
#pragma unroll
  for (int k = 0; k < KS; ++k) {
    int qx, qy;
    if (!fx_pos<FX_SX, L::SY, NW>(k, warp, lane, qx, qy)) continue;
    const int i = qy * FX_SX + qx;
    const i64* const A = qu + (qy + 2) * FX_UX + qx + 2;
    const i64* const B = A + L::UN;
    i64 ux = fx_c12(A[-2], A[-1], A[1], A[2]), vx = fx_c12(B[-2], B[-1], B[1], B[2]);
    i64 uy = fx_c12(A[-2 * FX_UX], A[-FX_UX], A[FX_UX], A[2 * FX_UX]);
    i64 vy = fx_c12(B[-2 * FX_UX], B[-FX_UX], B[FX_UX], B[2 * FX_UX]);
    const i64 mq = fx_from<58, false>(m[k], M);
    const FxSplit lf = fx_split(fx_from<58, false>(l[k], M)), mf = fx_split(mq), m2 = fx_split(mq << 1);
    i64 d, sh;
    if (edge) {  // closure rows (positions outside the grid are never read); sums of two may exceed 63 bits
      const int cx = zm_class(X0 - 2 + qx, n0), cy = zm_class(Y0 - 2 + qy, n1);
      if (cx != 4) {
        const i64* w = tw + 4 * cx;
        const int* o = to + 4 * cx;
        ux = fx_taps(w, A[o[0]], A[o[1]], A[o[2]], A[o[3]]);
        vx = fx_taps(w, B[o[0]], B[o[1]], B[o[2]], B[o[3]]);
      }
      if (cy != 4) {
        const i64* w = tw + 4 * cy;
        const int* o = to + 4 * cy;
        uy = fx_taps(w, A[o[0] * FX_UX], A[o[1] * FX_UX], A[o[2] * FX_UX], A[o[3] * FX_UX]);
        vy = fx_taps(w, B[o[0] * FX_UX], B[o[1] * FX_UX], B[o[2] * FX_UX], B[o[3] * FX_UX]);
      }
      d = fx_mulhi(lf, fx_split(ux)) + fx_mulhi(lf, fx_split(vy));
      sh = fx_mulhi(mf, fx_split(uy)) + fx_mulhi(mf, fx_split(vx));
    } else {
      d = fx_mulhi(lf, fx_split(ux + vy));
      sh = fx_mulhi(mf, fx_split(uy + vx));
    }
    sg[i] = d + fx_mulhi(m2, fx_split(ux));
    sg[L::SN + i] = d + fx_mulhi(m2, fx_split(vy));
    sg[2 * L::SN + i] = sh;
  }
  __syncthreads();
  // the tails of a source or a wave front reach down to the smallest FP64 numbers: their scale in two factors
  const int X1 = X < -900 ? -600 : 0;
  const double sc = s.kt144 * fx_pow2(X - X1), sc1 = fx_pow2(X1);
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    const int ty = warp + k * NW, y = Y0 + ty;
    if (!xu || y < g.off[1] || y >= g.off[1] + g.nu[1]) continue;
    const long long p = ro + o0 + ty * npx + lane;
    const i64* const XX = sg + (ty + 2) * FX_SX + lane + 2;
    const i64* const YY = XX + L::SN;
    const i64* const XY = YY + L::SN;
    i64 xx = fx_c12(XX[-2], XX[-1], XX[1], XX[2]), xy = fx_c12(XY[-2], XY[-1], XY[1], XY[2]);
    i64 yx = fx_c12(XY[-2 * FX_SX], XY[-FX_SX], XY[FX_SX], XY[2 * FX_SX]);
    i64 yy = fx_c12(YY[-2 * FX_SX], YY[-FX_SX], YY[FX_SX], YY[2 * FX_SX]);
    double k0, k1;
    if (edge) {
      const int cx = zm_class(x, n0), cy = zm_class(y, n1);
      double b0 = 0.0, b1 = 0.0;  // boundary terms of a free side: -D + H^{-1} B
      if (cx != 4) {
        const i64* w = tw + 4 * cx;
        const int* q = to + 4 * cx;
        xx = fx_taps(w, XX[q[0]], XX[q[1]], XX[q[2]], XX[q[3]]);
        xy = fx_taps(w, XY[q[0]], XY[q[1]], XY[q[2]], XY[q[3]]);
        if (x == 0) b0 = (double)fx_taps_one(s.bt, XX[0]), b1 = (double)fx_taps_one(s.bt, XY[0]);
        if (x == n0 - 1) b0 = -(double)fx_taps_one(s.bt, XX[0]), b1 = -(double)fx_taps_one(s.bt, XY[0]);
      }
      if (cy != 4) {
        const i64* w = tw + 4 * cy;
        const int* q = to + 4 * cy;
        yx = fx_taps(w, XY[q[0] * FX_SX], XY[q[1] * FX_SX], XY[q[2] * FX_SX], XY[q[3] * FX_SX]);
        yy = fx_taps(w, YY[q[0] * FX_SX], YY[q[1] * FX_SX], YY[q[2] * FX_SX], YY[q[3] * FX_SX]);
        if (y == 0) b0 += (double)fx_taps_one(s.bt, XY[0]), b1 += (double)fx_taps_one(s.bt, YY[0]);
        if (y == n1 - 1) b0 -= (double)fx_taps_one(s.bt, XY[0]), b1 -= (double)fx_taps_one(s.bt, YY[0]);
      }
      k0 = ((double)xx + (double)yx) + b0;
      k1 = ((double)xy + (double)yy) + b1;
    } else {
      k0 = (double)(xx + yx);
      k1 = (double)(xy + yy);
    }
    if (X1 != 0) k0 *= sc1, k1 *= sc1;
    const double cs = c[k] * sc;  // k0, k1 are +12 D sigma: -c dt^2 M^{-1} K u
    fx_update<MODE, FORCED>(f, p, u0[k], d0[k], a0[k], k0, cs, s);
    fx_update<MODE, FORCED>(f, p + F, u1[k], d1[k], a1[k], k1, cs, s);
  }
}

// ---- host side -----------------------------------------------------------------
const FxTaps& fx_table() {
  static const FxTaps t = [] {
    FxTaps q;
    int off[36];
    float unused[36];
    zm_class_taps(off, unused);
    static const int kCols[4][4] = {{0, 1, 2, 3}, {0, 2, -1, -1}, {0, 1, 3, 4}, {0, 2, 4, 5}};
    for (int c = 0; c < 9; ++c)
      for (int k = 0; k < 4; ++k) {
        double w;
        if (c == 4) {
          static const double iw[4] = {1.0, -8.0, 8.0, -1.0};
          w = iw[k];
        } else {
          const int r = c < 4 ? c : c - 5, j = kCols[r][k];
          w = j < 0 ? 0.0 : (c < 4 ? 12.0 : -12.0) * SBP_CLOSURE[r][j];
        }
        q.off[4 * c + k] = off[4 * c + k];
        q.w[4 * c + k] = (i64)(w * 0x1p57);
      }
    return q;
  }();
  static_assert(FX_TAP == 57, "scale of the table");
  return t;
}

template <int MODE, bool FORCED, int TY, int MINB>
cudaError_t fx_launch(const Geom& g, const WaveFields<double>& f, const FxStep& s, cudaStream_t st) {
  using L = Fx2<TY>;
  auto* k = step2d_o4_fx<MODE, FORCED, TY, MINB>;
  if (L::BYTES > 48 * 1024) {
    const cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)L::BYTES);
    if (e != cudaSuccess) return e;
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((g.nu[0] + s.shx + FX_TX - 1) / FX_TX, (g.nu[1] + s.shy + TY - 1) / TY, g.nrhs);
  cfg.blockDim = dim3(L::NT);
  cfg.dynamicSmemBytes = L::BYTES;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  const char* e = getenv("EWH_PDL");
  cfg.numAttrs = (e && e[0] == '0') ? 0 : 1;
  return cudaLaunchKernelEx(&cfg, k, g, f, s, fx_table());
}

template <int TY, int MINB>
cudaError_t fx_mode(const Geom& g, const WaveFields<double>& f, StepMode mode, FxStep& s, cudaStream_t st) {
  s.shx = zm_shift(g.nu[0], FX_TX, g.hi_free[0] != 0, 1);
  s.shy = zm_shift(g.nu[1], TY, g.hi_free[1] != 0, 1);
  const bool forced = f.frho != nullptr;
  switch (mode) {
    case STEP_FIRST:
      return forced ? fx_launch<STEP_FIRST, true, TY, MINB>(g, f, s, st)
                    : fx_launch<STEP_FIRST, false, TY, MINB>(g, f, s, st);
    case STEP_MID:
      return forced ? fx_launch<STEP_MID, true, TY, MINB>(g, f, s, st)
                    : fx_launch<STEP_MID, false, TY, MINB>(g, f, s, st);
    default:
      return forced ? fx_launch<STEP_LAST, true, TY, MINB>(g, f, s, st)
                    : fx_launch<STEP_LAST, false, TY, MINB>(g, f, s, st);
  }
}

}  // namespace

cudaError_t launch_fx2d(const Geom& g, int shape, const WaveFields<double>& f, StepMode mode, const StepScalars& sc,
                        cudaStream_t st) {
  if (g.dim != 2 || g.mapped) return cudaErrorInvalidValue;
  FxStep s{};
  s.kt = sc.kt;
  s.kt144 = sc.kt / 144.0;
  s.fc = sc.kt * sc.cosn;
  s.w0 = sc.w0;
  s.wnew = sc.wnew;
  s.bt = (i64)(12.0 * 48.0 / 17.0 * 0x1p57);
  switch (shape) {
    case 0: return fx_mode<16, 3>(g, f, mode, s, st);
    case 1: return fx_mode<8, 5>(g, f, mode, s, st);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace ewh
