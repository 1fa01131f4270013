// Order 2, 2D, small grids: all levels of a wave solve in one cooperative launch.
//
// A level of a small grid is latency, not work: at 62 x 62 nodes in FP64 the
// tiles of step2d_o2 take 3.7 us a level, of which the arithmetic of the whole grid
// is 0.3 us; the rest is the launch, its loads and an FP64 pipe that the CTAs
// share out badly.  Here every CTA keeps a tile of nodes for all levels:
// coefficients, delta and the filter's sum in registers (a thread per node and
// component), u in shared memory twice (a level reads one copy and writes the
// other, so one barrier per level is enough).  The tile's rim goes to the neighbours
// through L2: every 8-byte word carries 4 bytes of u and the level it belongs to,
// so a word that has arrived is its own flag and a level costs one store and one
// polled load of latency.  Two words of a slot alternate between levels; a
// CTA cannot be two levels ahead of a neighbour whose rim it needs.
//
// Per level, one right-hand side, against the tiles: 62 x 62 nodes 3.7 -> 1.6 us in
// FP64 and 1.4 -> 1.0 us in FP32, 150 x 150 5.8 -> 3.2 and 1.8 -> 1.4 us, 197 x 197 8.1 ->
// 4.9 and 1.9 -> 1.6 us.
// Bound by the store-to-poll latency through L2 and, in FP64, its pipe (20
// instructions a thread).  Grids that do not fit one CTA an SM keep the tiles.
//
// A solve whose waits give up ends with NaN.  In FP64, which right-hand sides, residuals and
// the solves that FP32 gave up on rest upon, a second launch then redoes it (step2d_o2_redo).
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>

#include "ewh_internal.cuh"
#include "ewh_order2.cuh"

namespace ewh {
namespace {

constexpr int S2_HEAD = 16;  // words before the rims (the error flag): a slot lies in one sector

struct Small2dShape {
  int px, nb, bx, by, P;  // CTAs along x and per rhs; nodes of a tile; threads per component
};

__device__ __forceinline__ unsigned long long s2_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
__device__ __forceinline__ unsigned s2_flag(const unsigned* p) {
  unsigned v;
  asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

// One value as words of 4 bytes and the tag: W words of 8 bytes (each a single access).
__device__ __forceinline__ void s2_send(unsigned long long* w, double v, unsigned tag) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(v), t = (unsigned long long)tag << 32;
  asm volatile("st.relaxed.gpu.global.v2.u64 [%0], {%1, %2};" ::"l"(w), "l"((b & 0xffffffffull) | t), "l"((b >> 32) | t)
               : "memory");
}
__device__ __forceinline__ void s2_send(unsigned long long* w, float v, unsigned tag) {
  const unsigned long long b = (unsigned long long)__float_as_uint(v) | ((unsigned long long)tag << 32);
  asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" ::"l"(w), "l"(b) : "memory");
}
__device__ __forceinline__ bool s2_take(const unsigned long long* w, unsigned tag, double& v) {
  unsigned long long a, b;
  asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];" : "=l"(a), "=l"(b) : "l"(w) : "memory");
  v = __longlong_as_double((long long)((a & 0xffffffffull) | (b << 32)));
  return (unsigned)(a >> 32) == tag && (unsigned)(b >> 32) == tag;
}
__device__ __forceinline__ bool s2_take(const unsigned long long* w, unsigned tag, float& v) {
  unsigned long long a;
  asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(a) : "l"(w) : "memory");
  v = __uint_as_float((unsigned)a);
  return (unsigned)(a >> 32) == tag;
}

// Wait for a slot of level `tag`: gives up after `lim` ns, 2^22 polls, or when another
// CTA raised the error flag (seen every 256 polls); a zero limit gives up at once.
// The CTA that gives up first counts the launch in bar[4].
template <typename T>
__device__ __forceinline__ bool s2_wait(const unsigned long long* w, unsigned tag, T& v, unsigned* err,
                                        unsigned* bar, unsigned long long lim) {
  bool ok = lim != 0ull;
  if (ok && s2_take(w, tag, v)) return true;
  const unsigned long long t0 = s2_ns();
  for (unsigned spins = 1; ok; ++spins) {
    if (s2_take(w, tag, v)) return true;
    if ((spins & 255u) == 0u) {
      if (s2_flag(err) != 0u) return false;
      ok = spins <= (1u << 22) && s2_ns() - t0 <= lim;
    }
  }
  if (atomicExch(err, 1u) == 0u) atomicAdd(bar + 4, 1u);
  return false;
}

// A node's row of K for one component in the form of the per-level kernels, times 2 h^2: axis a
// along the component, b across.  A free side takes the node itself for the neighbour that is
// missing, over half the width: offsets a0 .. b1 to the neighbours in an array of strides sx, sy.
template <typename T>
struct S2Node {
  O2Row<T> cf;
  int a0, a1, b0, b1;
  __device__ __forceinline__ S2Node(const Geom& g, const T* lam, const T* mu, int comp, int x, int y, int sx, int sy) {
    const long long pc = pidx(g, 0, 0, x, y, 0);
    const bool lox = x == 0, hix = x == g.n[0] - 1, loy = y == 0, hiy = y == g.n[1] - 1;
    const bool loa = comp ? loy : lox, hia = comp ? hiy : hix, lob = comp ? lox : loy, hib = comp ? hix : hiy;
    const int ga = comp ? g.np[0] : 1, gb = comp ? 1 : g.np[0];  // neighbours in the padded medium
    const int sa = comp ? sy : sx, sb = comp ? sx : sy;
    a0 = loa ? 0 : -sa, a1 = hia ? 0 : sa, b0 = lob ? 0 : -sb, b1 = hib ? 0 : sb;
    const T wa = loa || hia ? T(2) : T(1), wb = lob || hib ? T(2) : T(1);
    const T l0 = lam[pc], m0 = mu[pc], p0 = l0 + T(2) * m0;
    const long long qa0 = pc - (loa ? 0 : ga), qa1 = pc + (hia ? 0 : ga);
    const long long qb0 = pc - (lob ? 0 : gb), qb1 = pc + (hib ? 0 : gb);
    cf.ca0 = wa * (p0 + (lam[qa0] + T(2) * mu[qa0]));
    cf.ca1 = wa * (p0 + (lam[qa1] + T(2) * mu[qa1]));
    cf.cb0 = wb * (m0 + mu[qb0]);
    cf.cb1 = wb * (m0 + mu[qb1]);
    cf.la0 = T(0.5) * (loa ? T(-2) : wa) * wb * lam[qa0];
    cf.la1 = T(0.5) * (hia ? T(-2) : wa) * wb * lam[qa1];
    cf.mb0 = T(0.5) * (lob ? T(-2) : wb) * wa * mu[qb0];
    cf.mb1 = T(0.5) * (hib ? T(-2) : wb) * wa * mu[qb1];
  }
  // 2 h^2 rho M^{-1} K u; U the node's value, V that of the other component
  __device__ __forceinline__ T row(const T* U, const T* V, T u) const {
    return o2_row(cf, u, O2Vals<T>{U[a0], U[a1], U[b0], U[b1], V[a0 + b0], V[a0 + b1], V[a1 + b0], V[a1 + b1]});
  }
};

// NT_MAX: most threads of the CTA (512: no spills in FP64)
template <typename T, bool FORCED, int NT_MAX>
__global__ void __launch_bounds__(NT_MAX) step2d_o2_resident(Geom g, Small2dShape sh, Small2dIO<T> io) {
  if (g.dim != 2) return;
  constexpr int W = sizeof(T) / 4;  // words per value
  extern __shared__ double s2_smem[];
  T* const sb = reinterpret_cast<T*>(s2_smem);
  const unsigned long long lim = *reinterpret_cast<const unsigned long long*>(io.bar + 2);
  const int t = threadIdx.x, NT = blockDim.x;
  const int rhs = blockIdx.x / sh.nb, bid = blockIdx.x - rhs * sh.nb;
  const int nu0 = g.nu[0], nu1 = g.nu[1];
  const int X0 = (bid % sh.px) * sh.bx, Y0 = (bid / sh.px) * sh.by;  // first unknown of the tile
  const int wx = min(sh.bx, nu0 - X0), wy = min(sh.by, nu1 - Y0);
  const int SX = sh.bx + 2, TP = SX * (sh.by + 2), BUF = 2 * TP;
  for (int i = t; i < 2 * BUF; i += NT) sb[i] = T(0);
  __syncthreads();
  // u^0 on the tile and its ring (zero off the unknowns, in both copies)
  for (int i = t; i < BUF; i += NT) {
    const int c = i / TP, q = i - c * TP, ly = q / SX, lx = q - ly * SX;
    const int ux = X0 - 1 + lx, uy = Y0 - 1 + ly;
    if (lx < wx + 2 && ly < wy + 2 && ux >= 0 && ux < nu0 && uy >= 0 && uy < nu1)
      sb[i] = io.u0[pidx(g, rhs, c, ux + g.off[0], uy + g.off[1], 0)];
  }
  // the ring positions that this thread brings in: (component, position) pairs t and t + NT
  const int ring = 2 * (wx + 2) + 2 * wy;
  const long long half = (long long)g.nrhs * nu0 * nu1 * 2 * W;  // words per level parity
  unsigned* const err = reinterpret_cast<unsigned*>(io.xbuf);  // the launch's error flag, then the words
  unsigned long long* const xb = io.xbuf + S2_HEAD + (long long)rhs * nu0 * nu1 * 2 * W;
  int hdst[2] = {-1, -1}, hsrc[2] = {0, 0};
#pragma unroll
  for (int k = 0; k < 2; ++k) {
    const int i = t + k * NT;
    if (i < 2 * ring) {
      const int c = i >= ring, q = i - c * ring;
      int lx, ly;
      if (q < 2 * (wx + 2)) {
        ly = q < wx + 2 ? 0 : wy + 1;
        lx = q < wx + 2 ? q : q - (wx + 2);
      } else {
        const int r = q - 2 * (wx + 2);
        lx = r < wy ? 0 : wx + 1;
        ly = 1 + (r < wy ? r : r - wy);
      }
      const int ux = X0 - 1 + lx, uy = Y0 - 1 + ly;
      if (ux >= 0 && ux < nu0 && uy >= 0 && uy < nu1) {
        hdst[k] = c * TP + ly * SX + lx;
        hsrc[k] = ((uy * nu0 + ux) * 2 + c) * W;
      }
    }
  }
  // this thread's node and component (warps hold one component)
  const int comp = t >= sh.P, j = t - comp * sh.P;
  const int jx = j % sh.bx, jy = j / sh.bx;
  const bool own = jy < wy && jx < wx;
  const bool rim = own && (jx == 0 || jx == wx - 1 || jy == 0 || jy == wy - 1);
  const int ps = own ? (jy + 1) * SX + jx + 1 : SX + 1;
  const int x = X0 + (own ? jx : 0) + g.off[0], y = Y0 + (own ? jy : 0) + g.off[1];
  const long long pc = pidx(g, 0, 0, x, y, 0), p = pidx(g, rhs, comp, x, y, 0);
  const S2Node<T> nd(g, io.lam, io.mu, comp, x, y, 1, SX);
  const T ks = T(0.5 * io.kt) * io.irh2[pc], fr = FORCED ? io.frho[p] : T(0);
  const int oc = comp ? -TP : TP;  // to the other component
  __syncthreads();
  T uv = sb[comp * TP + ps], d = T(0), ac = o2_mul(T(io.w0), uv);
  unsigned long long* const xs =
      xb + ((long long)((Y0 + jy) * nu0 + (X0 + jx)) * 2 + comp) * W;
  bool alive = true;
  for (int n = 0; n < io.nsteps; ++n) {
    const T wn = T(__ldg(io.wnew + n)), kc = FORCED ? T((n == 0 ? 0.5 : 1.0) * io.kt * __ldg(io.cosn + n)) : T(0);
    T* const cur = sb + (n & 1) * BUF;
    if (n > 0) {
      bool bad = false;
#pragma unroll
      for (int k = 0; k < 2; ++k)
        if (hdst[k] >= 0) {
          T v = T(0);
          bad |= !s2_wait(xb + (n & 1) * half + hsrc[k], (unsigned)n, v, err, io.bar, lim);
          cur[hdst[k]] = v;
        }
      if (__syncthreads_or(bad)) {
        alive = false;
        break;
      }
    }
    if (own) {
      const T* const U = cur + comp * TP + ps;
      d = o2_delta<T, FORCED>(n == 0 ? T(0.5) * ks : ks, nd.row(U, U + oc, uv), kc, fr, d);
      const T un = o2_add(uv, d);
      if (n + 1 < io.nsteps) {
        if (rim) s2_send(xs + ((n + 1) & 1) * half, un, (unsigned)(n + 1));
        sb[((n + 1) & 1) * BUF + comp * TP + ps] = un;
      }
      ac = o2_fma(wn, un, ac);
      uv = un;
    }
  }
  if (own) io.acc[p] = alive ? ac : T(NAN);
}

// The solve again, level by level over the whole grid, by one CTA per right-hand side that
// waits for no other: the same bits, if a CTA of step2d_o2_resident gave up on a wait
// (else it returns at once; the launch costs 2.2 of 309 us at 62 x 62 nodes and 183 levels).
template <typename T, bool FORCED>
__global__ void __launch_bounds__(1024) step2d_o2_redo(Geom g, Small2dIO<T> io) {
  if (g.dim != 2 || *reinterpret_cast<const unsigned*>(io.xbuf) == 0u) return;
  const int nu0 = g.nu[0], N = nu0 * g.nu[1];
  for (int n = 0; n < io.nsteps; ++n) {
    const T* const cur = n & 1 ? io.u1 : io.u0;
    T* const next = n & 1 ? io.u0 : io.u1;
    const T wn = T(io.wnew[n]), kc = FORCED ? T((n == 0 ? 0.5 : 1.0) * io.kt * io.cosn[n]) : T(0);
    for (int i = threadIdx.x; i < 2 * N; i += blockDim.x) {
      const int comp = i >= N, j = i - comp * N, x = j % nu0 + g.off[0], y = j / nu0 + g.off[1];
      const long long p = pidx(g, blockIdx.x, comp, x, y, 0);
      const S2Node<T> nd(g, io.lam, io.mu, comp, x, y, 1, g.np[0]);
      const T ks = T(0.5 * io.kt) * io.irh2[pidx(g, 0, 0, x, y, 0)], fr = FORCED ? io.frho[p] : T(0);
      const T uv = cur[p], k = nd.row(cur + p, cur + p + (comp ? -g.field : g.field), uv);
      const T d = o2_delta<T, FORCED>(n == 0 ? T(0.5) * ks : ks, k, kc, fr, n == 0 ? T(0) : io.delta[p]);
      const T un = o2_add(uv, d);
      if (n + 1 < io.nsteps) next[p] = un, io.delta[p] = d;
      io.acc[p] = o2_fma(wn, un, n == 0 ? o2_mul(T(io.w0), uv) : io.acc[p]);
    }
    __syncthreads();
  }
}

template <typename T>
void (*small2d_kernel(int threads, bool forced))(Geom, Small2dShape, Small2dIO<T>) {
  if (forced) return threads <= 512 ? step2d_o2_resident<T, true, 512> : step2d_o2_resident<T, true, SMALL2D_THREADS>;
  return threads <= 512 ? step2d_o2_resident<T, false, 512> : step2d_o2_resident<T, false, SMALL2D_THREADS>;
}

}  // namespace

// Tiles for the current device: every CTA of the launch resident at once, the
// grid spread over all SMs; among those the least arithmetic on the busiest SM (in FP64
// its pipe takes 16 cycles an instruction of a warp), then the shortest ring.
template <typename T>
Small2dPlan plan_small2d(const Geom& g) {
  Small2dPlan best;
  if (g.dim != 2 || g.nrhs < 1 || g.nrhs > 4096 || g.mapped) return best;
  int dev = 0, sms = 0, coop = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev) != cudaSuccess || !coop) {
    cudaGetLastError();
    return best;
  }
  double best_cost = -1.0;
  const int nu0 = g.nu[0], nu1 = g.nu[1];
  for (int bx = 1; bx <= std::min(nu0, SMALL2D_THREADS / 2); ++bx)
    for (int by = 1; by <= std::min(nu1, SMALL2D_THREADS / 2 / bx); ++by) {
      const long long px = (nu0 + bx - 1) / bx, py = (nu1 + by - 1) / by, ctas = px * py * g.nrhs;
      if (ctas > sms) continue;
      const int P = (bx * by + 31) / 32 * 32, ring = 2 * (bx + 2) + 2 * by;
      const size_t smem = (size_t)4 * (bx + 2) * (by + 2) * sizeof(T);
      if (2 * ring > 4 * P || smem > 48 * 1024) continue;  // two ring values per thread
      const double cost = P / 32 * 2 * (sizeof(T) == 8 ? 20 * 16.0 : 40.0) + 2.0 * ring * 2;
      if (best_cost >= 0 && cost >= best_cost) continue;
      best_cost = cost;
      best = Small2dPlan{1, (int)px, (int)py, bx, by, P, smem};
    }
  for (int forced = 0; forced < 2 && best.ok; ++forced) {
    int per_sm = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, small2d_kernel<T>(2 * best.P, forced != 0), 2 * best.P,
                                                      best.smem) != cudaSuccess ||
        per_sm < 1) {
      cudaGetLastError();
      best.ok = 0;
    }
  }
  return best;
}

size_t small2d_words(const Geom& g, size_t elem) { return S2_HEAD + (size_t)g.nrhs * g.nu[0] * g.nu[1] * 4 * (elem / 4); }

template <typename T>
cudaError_t launch_small2d(const Geom& g, const Small2dPlan& p, const Small2dIO<T>& io, cudaStream_t st) {
  if (!p.ok || g.dim != 2 || io.nsteps < 1) return cudaErrorInvalidValue;
  // tag 0 is no level's: words of an earlier launch must not pass for this one's
  cudaError_t e = cudaMemsetAsync(io.xbuf, 0, small2d_words(g, sizeof(T)) * 8, st);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(p.px * p.py * g.nrhs);
  cfg.blockDim = dim3(2 * p.P);
  cfg.dynamicSmemBytes = p.smem;
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  e = cudaLaunchKernelEx(&cfg, small2d_kernel<T>(2 * p.P, io.frho != nullptr), g, Small2dShape{p.px, p.px * p.py, p.bx, p.by, p.P}, io);
  if (e != cudaSuccess || sizeof(T) == 4) return e;
  if (io.frho)
    step2d_o2_redo<T, true><<<g.nrhs, 1024, 0, st>>>(g, io);
  else
    step2d_o2_redo<T, false><<<g.nrhs, 1024, 0, st>>>(g, io);
  return cudaGetLastError();
}

template Small2dPlan plan_small2d<float>(const Geom&);
template Small2dPlan plan_small2d<double>(const Geom&);
template cudaError_t launch_small2d<float>(const Geom&, const Small2dPlan&, const Small2dIO<float>&, cudaStream_t);
template cudaError_t launch_small2d<double>(const Geom&, const Small2dPlan&, const Small2dIO<double>&, cudaStream_t);

}  // namespace ewh
