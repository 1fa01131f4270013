// 3x3 convolutions of the learned warm start (forward, data gradient, weight
// gradient) as implicit GEMMs on the 5th-generation tensor cores: operands by
// bulk-tensor (TMA) loads into swizzled shared memory, tcgen05.mma with the
// FP32 accumulators in tensor memory.  Activations NHWC, weights
// [Co][3][3][Ci], BF16 operands.
//
// A tile is a patch of 8 x 16 pixels (128 GEMM rows).  One image row of the
// patch is 8 pixels = one 8-row swizzle group, so the three vertical taps of
// a filter column are the same staged patch (18 image rows) read from a start
// address one group further: a patch is loaded once per horizontal tap (three
// times, not nine), and the zero padding of the convolution is the fill of
// the loads' out-of-range part.
//
// Waits on the barriers are bounded (one second); a CTA that gives up waits,
// bounded again, for its loads and MMAs in flight and writes NaN to its outputs.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <string>

#include "../../include/ewh.h"
#include "ewh_conv.cuh"
#include "ewh_internal.cuh"
#include "ewh_march.cuh"

namespace ewh {
namespace {

using bf16 = __nv_bfloat16;

constexpr int CV_PX = 8, CV_PY = 16;             // patch: pixels along x and y
constexpr int CV_ROWS = CV_PX * CV_PY;           // GEMM rows of a patch
constexpr int CV_HALO = CV_PX * (CV_PY + 2);     // staged pixels per horizontal tap
constexpr int CV_NT = 128;
constexpr int CV_STAGES_MAX = 4;
constexpr int CV_EPI = 32 * 20;                  // floats per warp of the epilogue's transpose (16 columns, padded)
constexpr float CV_LEAK = 0.1f;
constexpr int WG_PER = 8;                        // patches that one CTA of the weight gradient accumulates
constexpr unsigned long long CV_WAIT_NS = 1000000000ull;

// ---- PTX ---------------------------------------------------------------------
__device__ __forceinline__ bool cv_wait(uint64_t* bar, unsigned parity) {
  if (mbar_try(bar, parity)) return true;
  const unsigned long long t0 = zm_ns();
  while (!mbar_try(bar, parity))
    if (zm_ns() - t0 > CV_WAIT_NS) return false;
  return true;
}
__device__ __forceinline__ void cv_expect(uint64_t* bar, unsigned bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ void cv_load4(const CUtensorMap* m, unsigned dst, uint64_t* bar, int c0, int c1, int c2,
                                         int c3) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], "
      "[%6];" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(m)), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(smem_u32(bar))
      : "memory");
}
__device__ __forceinline__ void cv_load2(const CUtensorMap* m, unsigned dst, uint64_t* bar, int c0, int c1) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(
          dst),
      "l"(reinterpret_cast<uint64_t>(m)), "r"(c0), "r"(c1), "r"(smem_u32(bar))
      : "memory");
}
__device__ __forceinline__ void cv_commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
               : "memory");
}
__device__ __forceinline__ void cv_mma(unsigned d, uint64_t a, uint64_t b, unsigned idesc, bool acc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d),
      "l"(a), "l"(b), "r"(idesc), "r"((unsigned)acc)
      : "memory");
}
__device__ __forceinline__ void cv_ld16(unsigned taddr, float* v) {
  unsigned r[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, "
      "[%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}
__device__ __forceinline__ void cv_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void cv_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// Shared-memory matrix descriptor: start address, leading and stride byte
// offsets, layout (2, 4, 6: 128-, 64-, 32-byte swizzle).
__device__ __forceinline__ uint64_t cv_desc(unsigned addr, unsigned lbo, unsigned sbo, unsigned layout) {
  return (uint64_t)((addr & 0x3FFFFu) >> 4) | ((uint64_t)(lbo >> 4) << 16) | ((uint64_t)(sbo >> 4) << 32) |
         (1ull << 46) | ((uint64_t)layout << 61);
}
// Instruction descriptor: BF16 x BF16 -> FP32, M = 128, N columns; mn: both
// operands have the GEMM's M / N index contiguous (else its K index).
__host__ __device__ constexpr unsigned cv_idesc(int n, bool mn) {
  return (1u << 4) | (1u << 7) | (1u << 10) | (mn ? (3u << 15) : 0u) | ((unsigned)(n >> 3) << 17) | (8u << 24);
}

__device__ __forceinline__ void cv_tmem_alloc(unsigned* slot, int cols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(slot)), "r"(cols)
               : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void cv_tmem_free(unsigned t, int cols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(t), "r"(cols) : "memory");
}

struct CvBarriers {
  uint64_t full[CV_STAGES_MAX], empty[CV_STAGES_MAX], done;
  unsigned tmem;
  int issued, multiplied;  // K steps whose loads were requested, whose MMAs were issued: all, unless a wait gave up (noted
                           // there: a store after the loops slows the weight gradient by 4%)
};

// Barriers, tensor memory and the stage buffers of a CTA; returns the
// 1024-byte aligned shared address of stage 0.
__device__ __forceinline__ unsigned cv_begin(CvBarriers& b, unsigned char* raw, int cols, int steps) {
  if (threadIdx.x == 0) {
    for (int k = 0; k < CV_STAGES_MAX; ++k) {
      mbar_init(b.full + k, 1);
      mbar_init(b.empty + k, 1);
    }
    mbar_init(&b.done, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (threadIdx.x == 96) b.issued = b.multiplied = steps;
  if (threadIdx.x >= 64 && threadIdx.x < 96) cv_tmem_alloc(&b.tmem, cols);
  cv_fence_before();
  __syncthreads();
  cv_fence_after();
  return (smem_u32(raw) + 1023u) & ~1023u;
}
// The CTA's end; ok: this thread saw every MMA complete (else cv_drain's bounded waits first).
__device__ __forceinline__ void cv_end(CvBarriers& b, int cols, bool ok, int steps, int stages) {
  cv_fence_before();
  if (!__syncthreads_and(ok)) {
    if (threadIdx.x == 0)
      cv_drain(b.issued, b.multiplied, steps, stages, [&](CvBar kind, int stage, unsigned parity) {
        cv_wait(kind == CV_FULL ? b.full + stage : (kind == CV_EMPTY ? b.empty + stage : &b.done), parity);
      });
    __syncthreads();
  }
  if (threadIdx.x >= 64 && threadIdx.x < 96) cv_tmem_free(b.tmem, cols);
}

// ---------------------------------------------------------------------------
// Forward convolution (and, with flipped weights, the data gradient):
// y[pixel][co] = sum over taps and ci of x[pixel + tap][ci] w[co][tap][ci].
// GEMM per CTA: M = 128 pixels of a patch, N = BN output channels, K steps of
// (KC channels, one horizontal tap) = 3 vertical taps x KC / 16 MMAs.
//
// At 8 images of 256 x 256 x 32 the layer moves 134 MB (x, both outputs; 20 us
// at the copy rate) and takes 46 us, against 178 us for a 64 x 64 mma.sync tile with
// 16-wide K steps; at 64 x 64, 256 -> 128 channels 35 us (180 us), bound by the
// 260 MB that the CTAs load from L2.
// ---------------------------------------------------------------------------
struct ConvArgs {
  int N, H, W, Ci, Co;
  int tx, ty;           // patches per image along x and y
  int KC, rowb, layout; // channels per K step, bytes of a staged row, swizzle
  int BN, cols;         // output channels per CTA, tensor-memory columns
  int stages, a_bytes, b_bytes, stage_bytes;
  int act, vec;
  const float* bias;
  float* pre;
  bf16* out;
};

__global__ void __launch_bounds__(CV_NT) conv3x3_tc(const __grid_constant__ CUtensorMap mx,
                                                    const __grid_constant__ CUtensorMap mw, ConvArgs p) {
  extern __shared__ unsigned char cv_raw[];
  __shared__ CvBarriers bars;
  const int steps = 3 * (p.Ci / p.KC);
  const unsigned base = cv_begin(bars, cv_raw, p.cols, steps);
  const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
  const int tile = blockIdx.x;
  const int n = tile / (p.tx * p.ty), rem = tile - n * p.tx * p.ty;
  const int y0 = (rem / p.tx) * CV_PY, x0 = (rem % p.tx) * CV_PX;
  const int co0 = blockIdx.y * p.BN;
  const unsigned tmem = bars.tmem;
  if (t == 0) {  // loads: step = (channel block, horizontal tap)
    for (int s = 0; s < steps; ++s) {
      const int st = s % p.stages, c = (s / 3) * p.KC, kx = s % 3;
      if (s >= p.stages && !cv_wait(bars.empty + st, ((s / p.stages) - 1) & 1)) {
        bars.issued = s;
        break;
      }
      const unsigned a = base + st * p.stage_bytes, b = a + p.a_bytes;
      cv_expect(bars.full + st, p.a_bytes + 3 * p.b_bytes);
      cv_load4(&mx, a, bars.full + st, c, x0 + kx - 1, y0 - 1, n);
      for (int ky = 0; ky < 3; ++ky)
        cv_load2(&mw, b + ky * p.b_bytes, bars.full + st, (3 * ky + kx) * p.Ci + c, co0);
    }
  } else if (t == 32) {  // one thread issues the MMAs
    const unsigned idesc = cv_idesc(p.BN, false);
    for (int s = 0; s < steps; ++s) {
      const int st = s % p.stages;
      if (!cv_wait(bars.full + st, (s / p.stages) & 1)) {
        bars.multiplied = s;
        break;
      }
      cv_fence_after();
      const unsigned a = base + st * p.stage_bytes, b = a + p.a_bytes;
      for (int ky = 0; ky < 3; ++ky)
        for (int k = 0; k < p.KC; k += 16) {
          const uint64_t da = cv_desc(a + ky * CV_PX * p.rowb + 2 * k, 16, 8 * p.rowb, p.layout);
          const uint64_t db = cv_desc(b + ky * p.b_bytes + 2 * k, 16, 8 * p.rowb, p.layout);
          cv_mma(tmem, da, db, idesc, (s | ky | k) != 0);
        }
      cv_commit(s + 1 < steps ? bars.empty + st : &bars.done);
    }
  }
  __syncwarp();
  // epilogue: row = pixel; 16 columns at a time through a transpose in shared
  // memory (the stage buffers are free once the last MMA is done), so that
  // stores run along the channels of a pixel
  const bool ok = cv_wait(&bars.done, 0);
  cv_fence_after();
  __syncthreads();
  float* const tr = reinterpret_cast<float*>(cv_raw + (base - smem_u32(cv_raw))) + warp * CV_EPI;
  const float nanv = __int_as_float(0x7fc00000);
  for (int cb = 0; cb < p.BN && co0 + cb < p.Co; cb += 16) {
    float v[16];
    cv_ld16(tmem + ((unsigned)(warp * 32) << 16) + cb, v);
#pragma unroll
    for (int q = 0; q < 4; ++q)
      *reinterpret_cast<float4*>(tr + lane * 20 + 4 * q) = make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
    __syncwarp();
    const int co = co0 + cb + 4 * (lane & 3);
    float4 bi = make_float4(0.f, 0.f, 0.f, 0.f);
    if (p.bias && co < p.Co) bi = make_float4(p.bias[co], p.bias[co + 1], p.bias[co + 2], p.bias[co + 3]);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int r = 8 * i + (lane >> 2), row = warp * 32 + r;
      const int y = y0 + (row >> 3), x = x0 + (row & 7);
      if (y >= p.H || x >= p.W || co >= p.Co) continue;
      float4 s = *reinterpret_cast<const float4*>(tr + r * 20 + 4 * (lane & 3));
      s.x += bi.x, s.y += bi.y, s.z += bi.z, s.w += bi.w;
      if (!ok) s = make_float4(nanv, nanv, nanv, nanv);
      const long long o = (((long long)n * p.H + y) * p.W + x) * p.Co + co;
      if (p.pre) {
        if (p.vec) {
          *reinterpret_cast<float4*>(p.pre + o) = s;
        } else {
          p.pre[o] = s.x, p.pre[o + 1] = s.y, p.pre[o + 2] = s.z, p.pre[o + 3] = s.w;
        }
      }
      if (p.out) {
        if (p.act == 1) {
          s.x = s.x > 0.f ? s.x : CV_LEAK * s.x;
          s.y = s.y > 0.f ? s.y : CV_LEAK * s.y;
          s.z = s.z > 0.f ? s.z : CV_LEAK * s.z;
          s.w = s.w > 0.f ? s.w : CV_LEAK * s.w;
        }
        const __nv_bfloat162 lo = __floats2bfloat162_rn(s.x, s.y), hi = __floats2bfloat162_rn(s.z, s.w);
        if (p.vec) {
          uint2 u;
          u.x = *reinterpret_cast<const unsigned*>(&lo);
          u.y = *reinterpret_cast<const unsigned*>(&hi);
          *reinterpret_cast<uint2*>(p.out + o) = u;
        } else {
          p.out[o] = lo.x, p.out[o + 1] = lo.y, p.out[o + 2] = hi.x, p.out[o + 3] = hi.y;
        }
      }
    }
    __syncwarp();
  }
  cv_end(bars, p.cols, ok, steps, p.stages);
}

// ---------------------------------------------------------------------------
// Weight gradient: dw[co][tap][ci] = sum over pixels of dy[p][co] x[p + tap][ci].
// GEMM with the pixels as K: both operands have their channel index
// contiguous (M / N major).  M = 128 rows from x, N = NB output channels, a K
// step of 16 pixels = two image rows of a patch.
//   KC < 64: the 128 rows are 128 / KC blocks of KC channels, block j reading
//     the staged patch j image rows further down: the first three are the
//     vertical taps (the rest are unused rows), so one MMA per horizontal tap
//     covers three taps;
//   KC = 64: the rows are 128 channels, one MMA per vertical tap, the
//     horizontal tap is the CTA's.
// A CTA sums WG_PER patches and adds its part to dw with atomics: the tensor
// cores' FP32 accumulation truncates, so its error grows with the number of
// accumulated steps (relative 1.2e-6 at 64 steps of 16 pixels, 2.4e-6 at 128,
// measured on 524288 pixels against FP64); 1024 pixels keep it at the former.
// 37 us at 8 x 256 x 256, 32 -> 32 channels and 43 us at 8 x 64 x 64, 256 ->
// 128, against 1590 and 970 us for mma.sync on operands transposed element by
// element into shared memory.
// ---------------------------------------------------------------------------
struct WgradArgs {
  int N, H, W, Ci, Co;
  int tx, ty, patches;
  int KC, rowx, layx;       // x: channels per block, bytes of a row, swizzle
  int KO, rowo, layo;       // dy
  int NB, cols, cob;        // output channels per CTA, tensor-memory columns, blocks of output channels
  int x_copy;               // bytes of one staged x patch (one horizontal tap or channel block)
  int stages, o_bytes, stage_bytes, tx_bytes;
  int ragged;               // the patches cover more than the images
  const bf16 *x, *dy;
  float* dw;
};

// A pixel of a patch beyond the image is zero in dy, but it meets values inside the image in x: an
// infinity or a NaN there makes NaN of sums that the pixel does not belong to.  So
// sums that came out as NaN in images that the patches do not divide are formed again, one by
// one, over the pixels of the images.
__device__ float wgrad_plain(const WgradArgs& p, int q0, int steps, int co, int tap, int ci) {
  float s = 0.f;
  for (int q = q0; q < q0 + steps; ++q) {
    const int n = q / (p.tx * p.ty), rem = q - n * p.tx * p.ty;
    const int y0 = (rem / p.tx) * CV_PY, x0 = (rem % p.tx) * CV_PX;
    for (int i = 0; i < CV_ROWS; ++i) {
      const int y = y0 + i / CV_PX, x = x0 + i % CV_PX, yy = y + tap / 3 - 1, xx = x + tap % 3 - 1;
      if (y >= p.H || x >= p.W) continue;
      const bool in = yy >= 0 && yy < p.H && xx >= 0 && xx < p.W;  // the zero padding takes part
      const float a = in ? __bfloat162float(p.x[(((long long)n * p.H + yy) * p.W + xx) * p.Ci + ci]) : 0.f;
      s += __bfloat162float(p.dy[(((long long)n * p.H + y) * p.W + x) * p.Co + co]) * a;
    }
  }
  return s;
}
// The groups of 16 columns marked in `redo` (bit j 4 + column / 16) of this warp's rows, added to dw.
__device__ __noinline__ void wgrad_redo(const WgradArgs& p, unsigned redo, unsigned trow, int q0, int steps, int co0,
                                        int tap0, int dtap, int ci, bool live) {
  for (; redo; redo &= redo - 1) {
    const int bit = __ffs(redo) - 1, j = bit / 4, cb = bit % 4 * 16;
    float v[16];
    cv_ld16(trow + j * p.NB + cb, v);
    for (int i = 0; i < 16 && live; ++i) {
      const int co = co0 + cb + i, tap = tap0 + dtap * j;
      if (co >= p.Co) break;
      const float a = isnan(v[i]) ? wgrad_plain(p, q0, steps, co, tap, ci) : v[i];
      atomicAdd(p.dw + ((long long)co * 9 + tap) * p.Ci + ci, a);
    }
    __syncwarp();
  }
}

__global__ void __launch_bounds__(CV_NT) conv3x3_wgrad_tc(const __grid_constant__ CUtensorMap mx,
                                                          const __grid_constant__ CUtensorMap mo,
                                                          const __grid_constant__ WgradArgs p) {
  extern __shared__ unsigned char cv_raw[];
  __shared__ CvBarriers bars;
  const int q0 = blockIdx.x * WG_PER, steps = min(WG_PER, p.patches - q0);
  const unsigned base = cv_begin(bars, cv_raw, p.cols, steps);
  const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
  const bool wide = p.KC == 64;
  int blk = blockIdx.y;
  const int co0 = (blk % p.cob) * p.NB;
  blk /= p.cob;
  const int kxf = wide ? blk % 3 : 0;
  const int ci0 = wide ? (blk / 3) * 128 : blk * p.KC;
  const unsigned tmem = bars.tmem;
  if (t == 0) {
    for (int s = 0; s < steps; ++s) {
      const int st = s % p.stages;
      if (s >= p.stages && !cv_wait(bars.empty + st, ((s / p.stages) - 1) & 1)) {
        bars.issued = s;
        break;
      }
      const int q = q0 + s, n = q / (p.tx * p.ty), rem = q - n * p.tx * p.ty;
      const int y0 = (rem / p.tx) * CV_PY, x0 = (rem % p.tx) * CV_PX;
      const unsigned o = base + st * p.stage_bytes, x = o + p.o_bytes;
      cv_expect(bars.full + st, p.tx_bytes);
      for (int k = 0; k < p.NB; k += p.KO)
        cv_load4(&mo, o + (k / p.KO) * CV_ROWS * p.rowo, bars.full + st, co0 + k, x0, y0, n);
      if (wide) {
        for (int k = 0; k < 2; ++k)
          cv_load4(&mx, x + k * p.x_copy, bars.full + st, ci0 + 64 * k, x0 + kxf - 1, y0 - 1, n);
      } else {
        for (int kx = 0; kx < 3; ++kx) cv_load4(&mx, x + kx * p.x_copy, bars.full + st, ci0, x0 + kx - 1, y0 - 1, n);
      }
    }
  } else if (t == 32) {
    const unsigned idesc = cv_idesc(p.NB, true);
    const unsigned lbo = wide ? p.x_copy : 8 * p.rowx;       // between the blocks of M rows
    const unsigned off = wide ? 8 * p.rowx : p.x_copy;       // between the three MMAs of a K step
    for (int s = 0; s < steps; ++s) {
      const int st = s % p.stages;
      if (!cv_wait(bars.full + st, (s / p.stages) & 1)) {
        bars.multiplied = s;
        break;
      }
      cv_fence_after();
      const unsigned o = base + st * p.stage_bytes, x = o + p.o_bytes;
      for (int k = 0; k < CV_PY; k += 2) {
        const uint64_t db = cv_desc(o + k * 8 * p.rowo, CV_ROWS * p.rowo, 8 * p.rowo, p.layo);
        for (int j = 0; j < 3; ++j) {
          const uint64_t da = cv_desc(x + j * off + k * 8 * p.rowx, lbo, 8 * p.rowx, p.layx);
          cv_mma(tmem + j * p.NB, da, db, idesc, (s | k) != 0);
        }
      }
      cv_commit(s + 1 < steps ? bars.empty + st : &bars.done);
    }
  }
  __syncwarp();
  const bool ok = cv_wait(&bars.done, 0);
  cv_fence_after();
  // row m, column j NB + co: consecutive lanes are consecutive ci
  const int m = warp * 32 + lane;
  const int ci = ci0 + (wide ? m : m % p.KC), kyr = m / p.KC;
  const bool live = wide ? ci < p.Ci : kyr < 3;
  const int tap0 = wide ? kxf : 3 * kyr, dtap = wide ? 3 : 1;
  const unsigned trow = tmem + ((unsigned)(warp * 32) << 16);
  unsigned redo = 0;  // groups of columns left to wgrad_redo
  if (wide || warp * 32 < 3 * p.KC)
    for (int j = 0; j < 3; ++j) {
      const int tap = tap0 + dtap * j;
      for (int cb = 0; cb < p.NB && co0 + cb < p.Co; cb += 16) {
        float v[16];
        cv_ld16(trow + j * p.NB + cb, v);
        if (p.ragged && ok) {
          float s[8];
#pragma unroll
          for (int i = 0; i < 8; ++i) s[i] = v[i] + v[i + 8];
#pragma unroll
          for (int i = 0; i < 4; ++i) s[i] += s[i + 4];
          if (__any_sync(0xffffffffu, live && isnan((s[0] + s[1]) + (s[2] + s[3])))) {
            redo |= 1u << (4 * j + cb / 16);
            continue;
          }
        }
        if (live)
#pragma unroll
          for (int i = 0; i < 16; ++i)
            if (co0 + cb + i < p.Co)
              atomicAdd(p.dw + ((long long)(co0 + cb + i) * 9 + tap) * p.Ci + ci,
                        ok ? v[i] : __int_as_float(0x7fc00000));
        __syncwarp();
      }
    }
  if (redo) wgrad_redo(p, redo, trow, q0, steps, co0, tap0, dtap, ci, live);
  cv_end(bars, p.cols, ok, steps, p.stages);
}

// ---- host side ----------------------------------------------------------------
int block_of(int c) { return c % 64 == 0 ? 64 : (c % 32 == 0 ? 32 : 16); }
int layout_of(int kc) { return kc == 64 ? 2 : (kc == 32 ? 4 : 6); }
CUtensorMapSwizzle swizzle_of(int kc) {
  return kc == 64 ? CU_TENSOR_MAP_SWIZZLE_128B : (kc == 32 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_32B);
}
int columns_of(int n) {  // tensor-memory columns: a power of two, at least 32
  int c = 32;
  while (c < n) c *= 2;
  return c;
}

// Activations [N][H][W][C]: boxes of kc channels x 8 x rows pixels.
bool map_pixels(CUtensorMap* m, const void* x, int N, int H, int W, int C, int kc, int rows) {
  const cuuint64_t dims[4] = {(cuuint64_t)C, (cuuint64_t)W, (cuuint64_t)H, (cuuint64_t)N};
  const cuuint64_t strides[3] = {(cuuint64_t)C * 2, (cuuint64_t)W * C * 2, (cuuint64_t)H * W * C * 2};
  const cuuint32_t box[4] = {(cuuint32_t)kc, CV_PX, (cuuint32_t)rows, 1};
  const cuuint32_t es[4] = {1, 1, 1, 1};
  EncodeTiledFn enc = encode_fn();
  return enc && enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(x), dims, strides, box, es,
                    CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle_of(kc), CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                    CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}
// Weights [Co][9 Ci]: boxes of kc columns x bn rows.
bool map_weights(CUtensorMap* m, const void* w, int Ci, int Co, int kc, int bn) {
  const cuuint64_t dims[2] = {(cuuint64_t)9 * Ci, (cuuint64_t)Co};
  const cuuint64_t strides[1] = {(cuuint64_t)9 * Ci * 2};
  const cuuint32_t box[2] = {(cuuint32_t)kc, (cuuint32_t)bn};
  const cuuint32_t es[2] = {1, 1};
  EncodeTiledFn enc = encode_fn();
  return enc && enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(w), dims, strides, box, es,
                    CU_TENSOR_MAP_INTERLEAVE_NONE, swizzle_of(kc), CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                    CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Stages, shared memory of a CTA: up to `want` stages; at least so much that
// no more CTAs fit an SM than its 512 tensor-memory columns serve (an
// allocation would otherwise wait for another CTA to end).
constexpr int CV_SMEM_SM = 228 * 1024, CV_SMEM_CTA = 226 * 1024;
int shared_bytes(int stage_bytes, int want, int cols, int* stages) {
  int s = std::min(want, CV_STAGES_MAX);
  while (s > 1 && s * stage_bytes + 1024 > CV_SMEM_CTA) --s;
  *stages = s;
  const int least = CV_SMEM_SM / (512 / cols + 1) + 1;
  return std::max(std::max(s * stage_bytes, (int)(4 * CV_EPI * sizeof(float))) + 1024, std::min(least, CV_SMEM_CTA));
}

cudaError_t launch_err(bool ok) { return ok ? cudaGetLastError() : cudaErrorNotSupported; }

}  // namespace

// y = conv3x3(x, w) + bias; pre FP32 and / or out BF16 (leaky ReLU when act = 1).
cudaError_t launch_conv3x3(const void* x, const void* w, const float* bias, float* pre, void* out, int act, int N,
                           int H, int W, int Ci, int Co, cudaStream_t st) {
  ConvArgs p{};
  p.N = N, p.H = H, p.W = W, p.Ci = Ci, p.Co = Co;
  p.tx = (W + CV_PX - 1) / CV_PX;
  p.ty = (H + CV_PY - 1) / CV_PY;
  p.KC = block_of(Ci);
  p.rowb = 2 * p.KC;
  p.layout = layout_of(p.KC);
  // at most 64 output channels per CTA: two CTAs per SM, one storing while the
  // other multiplies
  p.BN = std::min(64, (Co + 15) / 16 * 16);
  p.cols = columns_of(p.BN);
  p.a_bytes = CV_HALO * p.rowb;
  p.b_bytes = p.BN * p.rowb;
  p.stage_bytes = (p.a_bytes + 3 * p.b_bytes + 1023) / 1024 * 1024;
  p.act = act;
  p.bias = bias;
  p.pre = pre;
  p.out = (bf16*)out;
  p.vec = ((uintptr_t)pre % 16 == 0 && (uintptr_t)out % 8 == 0) ? 1 : 0;
  // ahead of the tensor maps: a runtime call, which binds a context to a thread that has none
  cudaError_t e = cudaFuncSetAttribute(conv3x3_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, CV_SMEM_CTA);
  if (e != cudaSuccess) return e;
  CUtensorMap mx, mw;
  if (!map_pixels(&mx, x, N, H, W, Ci, p.KC, CV_PY + 2) || !map_weights(&mw, w, Ci, Co, p.KC, p.BN))
    return launch_err(false);
  const int bytes = shared_bytes(p.stage_bytes, std::min(3 * (Ci / p.KC), p.KC == 64 ? 2 : 3), p.cols, &p.stages);
  const dim3 grid((unsigned)((long long)N * p.tx * p.ty), (unsigned)((Co + p.BN - 1) / p.BN));
  conv3x3_tc<<<grid, CV_NT, bytes, st>>>(mx, mw, p);
  return launch_err(true);
}

// dw += the weight gradient (dw zeroed by the caller on the same stream).
cudaError_t launch_conv3x3_wgrad(const void* x, const void* dy, float* dw, int N, int H, int W, int Ci, int Co,
                                 cudaStream_t st) {
  WgradArgs p{};
  p.N = N, p.H = H, p.W = W, p.Ci = Ci, p.Co = Co;
  p.tx = (W + CV_PX - 1) / CV_PX;
  p.ty = (H + CV_PY - 1) / CV_PY;
  const long long patches = (long long)N * p.tx * p.ty;
  if (patches > 0x7fffffffLL) return cudaErrorInvalidValue;
  p.patches = (int)patches;
  p.KC = block_of(Ci);
  p.rowx = 2 * p.KC;
  p.layx = layout_of(p.KC);
  p.KO = block_of(Co);
  p.rowo = 2 * p.KO;
  p.layo = layout_of(p.KO);
  p.NB = std::min(64, Co);  // at most 192 accumulator columns: two CTAs per SM
  p.NB = p.NB / p.KO * p.KO;
  p.cob = (Co + p.NB - 1) / p.NB;
  p.cols = columns_of(3 * p.NB);
  const bool wide = p.KC == 64;
  p.x_copy = CV_HALO * p.rowx;
  p.o_bytes = CV_ROWS * p.rowo * (p.NB / p.KO);
  p.tx_bytes = p.o_bytes + (wide ? 2 : 3) * p.x_copy;
  // the unused M rows of the KC < 64 form read up to five image rows past the last patch
  p.stage_bytes = (p.tx_bytes + (wide ? 0 : 5 * 8 * p.rowx) + 1023) / 1024 * 1024;
  const int blocks = p.cob * (wide ? 3 * ((Ci + 127) / 128) : Ci / p.KC);
  const int bytes = shared_bytes(p.stage_bytes, 2, p.cols, &p.stages);
  p.ragged = W % CV_PX != 0 || H % CV_PY != 0;
  p.x = (const bf16*)x;
  p.dy = (const bf16*)dy;
  p.dw = dw;
  cudaError_t e = cudaFuncSetAttribute(conv3x3_wgrad_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, CV_SMEM_CTA);
  if (e != cudaSuccess) return e;  // before the maps, as above
  CUtensorMap mx, mo;
  if (!map_pixels(&mx, x, N, H, W, Ci, p.KC, CV_PY + 2) || !map_pixels(&mo, dy, N, H, W, Co, p.KO, CV_PY))
    return launch_err(false);
  const dim3 grid((unsigned)((p.patches + WG_PER - 1) / WG_PER), (unsigned)blocks);
  conv3x3_wgrad_tc<<<grid, CV_NT, bytes, st>>>(mx, mo, p);
  return launch_err(true);
}

}  // namespace ewh
