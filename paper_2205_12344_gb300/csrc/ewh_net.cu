// Layers of the learned warm start (a small convolutional encoder-decoder that
// maps medium, forcing and frequency to an initial guess for the CG solve of
// M (I - S) v = M Pi 0): the entry points of the 3x3 convolutions and their
// gradients (kernels in ewh_conv.cu) and the small element-wise layers.  Activations are NHWC with channel counts that are
// multiples of 16; weights are [Co][3][3][Ci].  The paper has no learned part:
// these kernels serve the precision/warm-start forms of the solver.
#include <cooperative_groups.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <string>

#include "../../include/ewh.h"
#include "ewh_conv.cuh"
#include "ewh_internal.cuh"

namespace {

using bf16 = __nv_bfloat16;

constexpr float LEAK = 0.1f;

// weights [Co][3][3][Ci] -> flipped/transposed [Ci][3][3][Co] (for the data gradient)
__global__ void flip_transpose_kernel(const bf16* __restrict__ w, bf16* __restrict__ wt, int Ci, int Co) {
  const long long total = (long long)Co * 9 * Ci;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total; i += (long long)gridDim.x * blockDim.x) {
    const int ci = (int)(i % Ci);
    const int k = (int)((i / Ci) % 9);
    const int co = (int)(i / (9LL * Ci));
    const int ky = k / 3, kx = k % 3;
    wt[(((long long)ci * 3 + (2 - ky)) * 3 + (2 - kx)) * Co + co] = w[i];
  }
}

// ---------------------------------------------------------------------------
// Weight gradient of operands that the bulk-tensor loads of ewh_conv.cu cannot
// address (x or dy off a 16-byte boundary): element-wise loads, mma.sync.
// dw[co][ky][kx][ci] = sum_p dy[p][co] x[p shifted][ci].
// CTA: 64 co x 64 ci for one (ky, kx) and one chunk of pixels (split K);
// partial sums are added into the FP32 result with atomics.  A = dy^T (co x
// pixels), B = shifted x (pixels x ci), K step = 16 pixels.  Bound by its scalar
// staging: 1590 us at 8 x 256 x 256, 32 -> 32 channels (37 us aligned), 970 us at
// 8 x 64 x 64, 256 -> 128 (43 us).
// ---------------------------------------------------------------------------
// D (16x8 f32) += A (16x16 bf16, row) * B (16x8 bf16, col)
__device__ __forceinline__ void mma_bf16_16816(float* d, const unsigned* a, const unsigned* b) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 "
      "{%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};\n"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

__device__ __forceinline__ unsigned ld32(const bf16* p) { return *reinterpret_cast<const unsigned*>(p); }

constexpr int WG_PIX_CHUNK = 1024, WG_LD = 24;  // LD: padded row length (bf16)

__global__ void __launch_bounds__(128) conv3x3_wgrad_unaligned(const bf16* __restrict__ x, const bf16* __restrict__ dy,
                                                            float* __restrict__ dw, int N, int H, int W, int Ci,
                                                            int Co) {
  __shared__ __align__(16) bf16 sA[64][WG_LD];  // [co][pixel]
  __shared__ __align__(16) bf16 sB[64][WG_LD];  // [ci][pixel]
  const int k9 = blockIdx.x % 9;
  const int ky = k9 / 3, kx = k9 % 3;
  const int ci_tiles = (Ci + 63) / 64;
  const int co0 = (blockIdx.x / 9 / ci_tiles) * 64;
  const int ci0 = ((blockIdx.x / 9) % ci_tiles) * 64;
  const long long P = (long long)N * H * W;
  const long long p_begin = (long long)blockIdx.y * WG_PIX_CHUNK;
  const long long p_end = p_begin + WG_PIX_CHUNK < P ? p_begin + WG_PIX_CHUNK : P;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int gid = lane >> 2, tig = lane & 3;
  // warp tile: 16 co (rows) x 64 ci (8 n-tiles)
  float acc[8][4];
#pragma unroll
  for (int j = 0; j < 8; ++j)
#pragma unroll
    for (int q = 0; q < 4; ++q) acc[j][q] = 0.f;
  for (long long pb = p_begin; pb < p_end; pb += 16) {
    // stage dy[p][co0..co0+63] transposed into sA[co][p], and the shifted x
    for (int i = tid; i < 16 * 64; i += 128) {
      const int pl = i / 64, c = i % 64;
      const long long p = pb + pl;
      bf16 vdy = __float2bfloat16(0.f), vx = __float2bfloat16(0.f);
      if (p < p_end) {
        if (co0 + c < Co) vdy = dy[p * Co + co0 + c];
        const int n = (int)(p / ((long long)H * W));
        const int r = (int)(p - (long long)n * H * W);
        const int yy = r / W + ky - 1, xx = r % W + kx - 1;
        if (ci0 + c < Ci && yy >= 0 && yy < H && xx >= 0 && xx < W)
          vx = x[(((long long)n * H + yy) * W + xx) * Ci + ci0 + c];
      }
      sA[c][pl] = vdy;
      sB[c][pl] = vx;
    }
    __syncthreads();
    unsigned a[4];
    const int r0 = warp * 16 + gid;
    a[0] = ld32(&sA[r0][tig * 2]);
    a[1] = ld32(&sA[r0 + 8][tig * 2]);
    a[2] = ld32(&sA[r0][tig * 2 + 8]);
    a[3] = ld32(&sA[r0 + 8][tig * 2 + 8]);
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      unsigned b[2];
      b[0] = ld32(&sB[j * 8 + gid][tig * 2]);
      b[1] = ld32(&sB[j * 8 + gid][tig * 2 + 8]);
      mma_bf16_16816(acc[j], a, b);
    }
    __syncthreads();
  }
#pragma unroll
  for (int j = 0; j < 8; ++j)
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int co = co0 + warp * 16 + gid + (q >= 2 ? 8 : 0);
      const int ci = ci0 + j * 8 + tig * 2 + (q & 1);
      if (co < Co && ci < Ci) atomicAdd(&dw[(((long long)co * 3 + ky) * 3 + kx) * Ci + ci], acc[j][q]);
    }
}

// ---------------------------------------------------------------------------
// Element-wise layers
// ---------------------------------------------------------------------------
// db[c] = sum over pixels of dy[p][c].  A cluster of CTAs takes 8 channels (one
// 32-byte sector of every pixel), each CTA every gridDim.y-th run of 128 pixels;
// its first CTA adds the others' sums from their shared memory, in rank order,
// so the result does not depend on timing.  Bound by memory: one block per channel
// read each sector 8 times on 32 SMs (267 us for 524288 x 32; this one 20 us).
constexpr int BG_THREADS = 1024, BG_CH = 8, BG_PIX = BG_THREADS / BG_CH;
constexpr int BG_CLUSTER = 16;           // CTAs per cluster for long sums
constexpr long long BG_LONG = 16384;     // pixels from which the cluster pays
__global__ void __launch_bounds__(BG_THREADS) bias_grad_kernel(const float* __restrict__ dy, float* __restrict__ db,
                                                               long long P, int C) {
  __shared__ float warp_part[BG_THREADS / 32][BG_CH];
  __shared__ float cta_part[BG_CH];
  const int c0 = blockIdx.x * BG_CH, c = c0 + (int)(threadIdx.x % BG_CH);
  float s = 0.f;
  if (c < C) {
    const long long step = (long long)gridDim.y * BG_PIX;
    long long p = (long long)blockIdx.y * BG_PIX + threadIdx.x / BG_CH;
    const float* q = dy + p * C + c;
    for (; p + 7 * step < P; p += 8 * step, q += 8 * step * C) {  // eight loads in flight
      float v[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) v[k] = __ldg(q + k * step * C);
      s += ((v[0] + v[1]) + (v[2] + v[3])) + ((v[4] + v[5]) + (v[6] + v[7]));
    }
    for (; p < P; p += step, q += step * C) s += __ldg(q);
  }
  s += __shfl_xor_sync(0xffffffffu, s, 16);
  s += __shfl_xor_sync(0xffffffffu, s, 8);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (lane < BG_CH) warp_part[warp][lane] = s;
  __syncthreads();
  if (threadIdx.x < BG_CH) {
    float t = 0.f;
    for (int w = 0; w < BG_THREADS / 32; ++w) t += warp_part[w][threadIdx.x];
    cta_part[threadIdx.x] = t;
  }
  namespace cg = cooperative_groups;
  cg::cluster_group cl = cg::this_cluster();
  cl.sync();
  if (cl.block_rank() == 0 && threadIdx.x < BG_CH && c0 + (int)threadIdx.x < C) {
    float t = 0.f;
    for (unsigned r = 0; r < cl.num_blocks(); ++r) t += cl.map_shared_rank(cta_part, r)[threadIdx.x];
    db[c0 + threadIdx.x] = t;
  }
  cl.sync();  // the other CTAs' shared memory stays until it is read
}

__device__ __forceinline__ float leaky_grad(float pre, float dy) { return pre > 0.f ? dy : LEAK * dy; }

// vec: every pointer 16-byte (8-byte for the BF16 one) aligned; four values a
// thread and pass then (bound by memory: 14 bytes a value)
__global__ void leaky_bwd_kernel(const float* __restrict__ pre, const float* __restrict__ dy, float* __restrict__ dx,
                                 bf16* __restrict__ dx_bf, long long n, int vec) {
  const long long t = blockIdx.x * (long long)blockDim.x + threadIdx.x, nt = (long long)gridDim.x * blockDim.x;
  const long long n4 = vec ? n / 4 : 0;
  for (long long i = t; i < n4; i += nt) {
    const float4 a = __ldcs(reinterpret_cast<const float4*>(pre) + i), d = __ldcs(reinterpret_cast<const float4*>(dy) + i);
    const float4 g = make_float4(leaky_grad(a.x, d.x), leaky_grad(a.y, d.y), leaky_grad(a.z, d.z), leaky_grad(a.w, d.w));
    if (dx) reinterpret_cast<float4*>(dx)[i] = g;
    if (dx_bf) {
      const __nv_bfloat162 lo = __floats2bfloat162_rn(g.x, g.y), hi = __floats2bfloat162_rn(g.z, g.w);
      uint2 u;
      u.x = *reinterpret_cast<const unsigned*>(&lo);
      u.y = *reinterpret_cast<const unsigned*>(&hi);
      reinterpret_cast<uint2*>(dx_bf)[i] = u;
    }
  }
  for (long long i = 4 * n4 + t; i < n; i += nt) {
    const float g = leaky_grad(pre[i], dy[i]);
    if (dx) dx[i] = g;
    if (dx_bf) dx_bf[i] = __float2bfloat16(g);
  }
}

// NHWC 2x2 average pooling (bf16 in/out) and its gradient (f32)
__global__ void avgpool2_kernel(const bf16* __restrict__ x, bf16* __restrict__ y, int N, int H, int W, int C) {
  const int Ho = H / 2, Wo = W / 2;
  const long long total = (long long)N * Ho * Wo * C;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total; i += (long long)gridDim.x * blockDim.x) {
    const int c = (int)(i % C);
    const long long q = i / C;
    const int xo = (int)(q % Wo), yo = (int)((q / Wo) % Ho), n = (int)(q / ((long long)Wo * Ho));
    const long long b = (((long long)n * H + 2 * yo) * W + 2 * xo) * C + c;
    const float s = __bfloat162float(x[b]) + __bfloat162float(x[b + C]) + __bfloat162float(x[b + (long long)W * C]) +
                    __bfloat162float(x[b + (long long)W * C + C]);
    y[i] = __float2bfloat16(0.25f * s);
  }
}
__global__ void avgpool2_bwd_kernel(const float* __restrict__ dy, float* __restrict__ dx, int N, int H, int W, int C) {
  const long long total = (long long)N * H * W * C;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total; i += (long long)gridDim.x * blockDim.x) {
    const int c = (int)(i % C);
    const long long q = i / C;
    const int xx = (int)(q % W), yy = (int)((q / W) % H), n = (int)(q / ((long long)W * H));
    dx[i] = 0.25f * dy[(((long long)n * (H / 2) + yy / 2) * (W / 2) + xx / 2) * C + c];
  }
}
// nearest 2x upsampling of x[N,H,W,C] into channels [c_off, c_off + C) of y[N,2H,2W,Cy]
__global__ void upsample2_kernel(const bf16* __restrict__ x, bf16* __restrict__ y, int N, int H, int W, int C, int Cy,
                                 int c_off) {
  const long long total = (long long)N * 2 * H * 2 * W * C;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total; i += (long long)gridDim.x * blockDim.x) {
    const int c = (int)(i % C);
    const long long q = i / C;
    const int xx = (int)(q % (2 * W)), yy = (int)((q / (2 * W)) % (2 * H)), n = (int)(q / (4LL * W * H));
    y[(((long long)n * 2 * H + yy) * 2 * W + xx) * Cy + c_off + c] = x[(((long long)n * H + yy / 2) * W + xx / 2) * C + c];
  }
}
// gradient of upsample2 from channels [c_off, c_off + C) of dy[N,2H,2W,Cy]
__global__ void upsample2_bwd_kernel(const float* __restrict__ dy, float* __restrict__ dx, int N, int H, int W, int C,
                                     int Cy, int c_off) {
  const long long total = (long long)N * H * W * C;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total; i += (long long)gridDim.x * blockDim.x) {
    const int c = (int)(i % C);
    const long long q = i / C;
    const int xx = (int)(q % W), yy = (int)((q / W) % H), n = (int)(q / ((long long)W * H));
    float s = 0.f;
    for (int dyy = 0; dyy < 2; ++dyy)
      for (int dxx = 0; dxx < 2; ++dxx)
        s += dy[(((long long)n * 2 * H + 2 * yy + dyy) * 2 * W + 2 * xx + dxx) * Cy + c_off + c];
    dx[i] = s;
  }
}
// copy x[N,H,W,C] into channels [c_off, c_off + C) of y[N,H,W,Cy] (concatenation)
__global__ void copy_channels_kernel(const bf16* __restrict__ x, bf16* __restrict__ y, long long P, int C, int Cy,
                                     int c_off) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < P * C; i += (long long)gridDim.x * blockDim.x)
    y[(i / C) * Cy + c_off + (i % C)] = x[i];
}
// dx[p][c] (+)= dy[p][c_off + c]  (gradient of a concatenation slice)
__global__ void slice_channels_kernel(const float* __restrict__ dy, float* __restrict__ dx, long long P, int C, int Cy,
                                      int c_off, int accumulate) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < P * C; i += (long long)gridDim.x * blockDim.x) {
    const float v = dy[(i / C) * Cy + c_off + (i % C)];
    dx[i] = accumulate ? dx[i] + v : v;
  }
}
__global__ void f32_to_bf16_kernel(const float* __restrict__ a, bf16* __restrict__ b, long long n) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x)
    b[i] = __float2bfloat16(a[i]);
}
// Adam (Kingma and Ba 2015) with bias correction; also refreshes the BF16 copy
__global__ void adam_kernel(float* __restrict__ p, const float* __restrict__ g, float* __restrict__ m,
                            float* __restrict__ v, bf16* __restrict__ p_bf, long long n, float lr, float b1, float b2,
                            float eps, float c1, float c2) {
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.f - b1) * gi;
    const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    const float pi = p[i] - lr * (mi / c1) / (sqrtf(vi / c2) + eps);
    p[i] = pi;
    if (p_bf) p_bf[i] = __float2bfloat16(pi);
  }
}

// Per-sample scaled L2 loss on the first `cu` of `c` channels:
//   loss_s = 1/2 ||y_s - t_s||^2 / ||t_s||^2,  grad = (y - t) / (||t_s||^2 * nsamp)
// (t is FP32 [N][P][cu], y FP32 [N][P][c]); one block per sample.
__global__ void scaled_l2_kernel(const float* __restrict__ y, const float* __restrict__ t, float* __restrict__ grad,
                                 float* __restrict__ loss, long long P, int c, int cu, int nsamp) {
  __shared__ float s_tt[256], s_dd[256];
  const int n = blockIdx.x;
  const float* yn = y + (long long)n * P * c;
  const float* tn = t + (long long)n * P * cu;
  float tt = 0.f, dd = 0.f;
  for (long long i = threadIdx.x; i < P * cu; i += 256) {
    const float d = yn[(i / cu) * c + (i % cu)] - tn[i];
    tt += tn[i] * tn[i];
    dd += d * d;
  }
  s_tt[threadIdx.x] = tt;
  s_dd[threadIdx.x] = dd;
  __syncthreads();
  for (int o = 128; o > 0; o >>= 1) {
    if (threadIdx.x < o) {
      s_tt[threadIdx.x] += s_tt[threadIdx.x + o];
      s_dd[threadIdx.x] += s_dd[threadIdx.x + o];
    }
    __syncthreads();
  }
  const float inv = 1.f / fmaxf(s_tt[0], 1e-30f);
  if (threadIdx.x == 0) loss[n] = 0.5f * s_dd[0] * inv;
  float* gn = grad + (long long)n * P * c;
  for (long long i = threadIdx.x; i < P * c; i += 256) {
    const int ch = (int)(i % c);
    gn[i] = ch < cu ? (yn[i] - tn[(i / c) * cu + ch]) * inv / nsamp : 0.f;
  }
}

int egrid(long long n) {
  long long b = (n + 255) / 256;
  if (b > 4096) b = 4096;
  return (int)(b < 1 ? 1 : b);
}

bool aligned16(const void* p) { return (uintptr_t)p % 16 == 0; }

ewh_status nfail(const char* msg) {
  ewh::set_global_error(msg);
  return EWH_EINVAL;
}

ewh_status launched(cudaError_t e = cudaSuccess) {
  const cudaError_t pending = cudaGetLastError();
  if (e == cudaSuccess) e = pending;
  if (e != cudaSuccess) {
    ewh::set_global_error(std::string("warm-start kernel launch failed: ") + cudaGetErrorString(e));
    return EWH_ECUDA;
  }
  return EWH_OK;
}

}  // namespace

extern "C" {

ewh_status ewh_conv3x3_fwd(const void* x, const void* w, const float* bias, float* y_pre, void* y_act, int act, int N,
                           int H, int W, int Ci, int Co, void* stream) {
  if (!x || !w || (!y_pre && !y_act) || N < 1 || H < 1 || W < 1 || Ci < 16 || Ci % 16 || Co < 8 || Co % 8)
    return nfail("ewh_conv3x3_fwd: bad arguments (Ci multiple of 16, Co multiple of 8)");
  if (!aligned16(x) || !aligned16(w)) return nfail("ewh_conv3x3_fwd: x and w must be 16-byte aligned");
  return launched(ewh::launch_conv3x3(x, w, bias, y_pre, y_act, act, N, H, W, Ci, Co, (cudaStream_t)stream));
}

ewh_status ewh_conv3x3_dgrad(const void* dy, const void* w, void* w_scratch, float* dx, int N, int H, int W, int Ci,
                             int Co, void* stream) {
  if (!dy || !w || !w_scratch || !dx || Ci % 16 || Co % 16 || Ci < 16 || Co < 16)
    return nfail("ewh_conv3x3_dgrad: bad arguments (Ci, Co multiples of 16)");
  if (!aligned16(dy) || !aligned16(w_scratch)) return nfail("ewh_conv3x3_dgrad: dy and w_scratch must be 16-byte aligned");
  cudaStream_t st = (cudaStream_t)stream;
  flip_transpose_kernel<<<egrid(9LL * Ci * Co), 256, 0, st>>>((const bf16*)w, (bf16*)w_scratch, Ci, Co);
  return launched(ewh::launch_conv3x3(dy, w_scratch, nullptr, dx, nullptr, 0, N, H, W, Co, Ci, st));
}

ewh_status ewh_conv3x3_wgrad(const void* x, const void* dy, float* dw, int N, int H, int W, int Ci, int Co,
                             void* stream) {
  if (!x || !dy || !dw || Ci % 16 || Co % 16 || Ci < 16 || Co < 16)
    return nfail("ewh_conv3x3_wgrad: bad arguments (Ci, Co multiples of 16)");
  cudaStream_t st = (cudaStream_t)stream;
  const cudaError_t e = cudaMemsetAsync(dw, 0, sizeof(float) * 9LL * Ci * Co, st);
  if (e != cudaSuccess) return launched(e);
  if (!aligned16(x) || !aligned16(dy)) {
    const long long P = (long long)N * H * W;
    const int ci_t = (Ci + 63) / 64, co_t = (Co + 63) / 64;
    const dim3 grid((unsigned)(9 * ci_t * co_t), (unsigned)((P + WG_PIX_CHUNK - 1) / WG_PIX_CHUNK));
    conv3x3_wgrad_unaligned<<<grid, 128, 0, st>>>((const bf16*)x, (const bf16*)dy, dw, N, H, W, Ci, Co);
    return launched();
  }
  return launched(ewh::launch_conv3x3_wgrad(x, dy, dw, N, H, W, Ci, Co, st));
}

ewh_status ewh_bias_grad(const float* dy, float* db, long long P, int C, void* stream) {
  if (!dy || !db || P < 1 || C < 1) return nfail("ewh_bias_grad: bad arguments");
  const int cs = P >= BG_LONG ? BG_CLUSTER : 1;
  cudaError_t e = cudaFuncSetAttribute(bias_grad_kernel, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  if (e != cudaSuccess) return launched(e);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)((C + BG_CH - 1) / BG_CH), (unsigned)cs);
  cfg.blockDim = dim3(BG_THREADS);
  cfg.stream = (cudaStream_t)stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 1;
  attr[0].val.clusterDim.y = cs;
  attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return launched(cudaLaunchKernelEx(&cfg, bias_grad_kernel, dy, db, P, C));
}

ewh_status ewh_leaky_relu_bwd(const float* pre, const float* dy, float* dx, void* dx_bf16, long long n, void* stream) {
  if (!pre || !dy || (!dx && !dx_bf16) || n < 0) return nfail("ewh_leaky_relu_bwd: bad arguments");
  const int vec = ((uintptr_t)pre | (uintptr_t)dy | (uintptr_t)dx) % 16 == 0 && (uintptr_t)dx_bf16 % 8 == 0;
  leaky_bwd_kernel<<<egrid(vec ? n / 4 : n), 256, 0, (cudaStream_t)stream>>>(pre, dy, dx, (bf16*)dx_bf16, n, vec);
  return launched();
}

ewh_status ewh_avgpool2(const void* x, void* y, int N, int H, int W, int C, void* stream) {
  if (!x || !y || H % 2 || W % 2) return nfail("ewh_avgpool2: bad arguments (H, W even)");
  avgpool2_kernel<<<egrid((long long)N * H * W * C / 4), 256, 0, (cudaStream_t)stream>>>((const bf16*)x, (bf16*)y, N,
                                                                                          H, W, C);
  return launched();
}

ewh_status ewh_avgpool2_bwd(const float* dy, float* dx, int N, int H, int W, int C, void* stream) {
  if (!dy || !dx || H % 2 || W % 2) return nfail("ewh_avgpool2_bwd: bad arguments (H, W even)");
  avgpool2_bwd_kernel<<<egrid((long long)N * H * W * C), 256, 0, (cudaStream_t)stream>>>(dy, dx, N, H, W, C);
  return launched();
}

ewh_status ewh_upsample2(const void* x, void* y, int N, int H, int W, int C, int Cy, int c_off, void* stream) {
  if (!x || !y || c_off < 0 || c_off + C > Cy) return nfail("ewh_upsample2: bad arguments");
  upsample2_kernel<<<egrid(4LL * N * H * W * C), 256, 0, (cudaStream_t)stream>>>((const bf16*)x, (bf16*)y, N, H, W, C,
                                                                                  Cy, c_off);
  return launched();
}

ewh_status ewh_upsample2_bwd(const float* dy, float* dx, int N, int H, int W, int C, int Cy, int c_off, void* stream) {
  if (!dy || !dx || c_off < 0 || c_off + C > Cy) return nfail("ewh_upsample2_bwd: bad arguments");
  upsample2_bwd_kernel<<<egrid((long long)N * H * W * C), 256, 0, (cudaStream_t)stream>>>(dy, dx, N, H, W, C, Cy,
                                                                                           c_off);
  return launched();
}

ewh_status ewh_copy_channels(const void* x, void* y, long long P, int C, int Cy, int c_off, void* stream) {
  if (!x || !y || c_off < 0 || c_off + C > Cy) return nfail("ewh_copy_channels: bad arguments");
  copy_channels_kernel<<<egrid(P * C), 256, 0, (cudaStream_t)stream>>>((const bf16*)x, (bf16*)y, P, C, Cy, c_off);
  return launched();
}

ewh_status ewh_slice_channels(const float* dy, float* dx, long long P, int C, int Cy, int c_off, int accumulate,
                              void* stream) {
  if (!dy || !dx || c_off < 0 || c_off + C > Cy) return nfail("ewh_slice_channels: bad arguments");
  slice_channels_kernel<<<egrid(P * C), 256, 0, (cudaStream_t)stream>>>(dy, dx, P, C, Cy, c_off, accumulate);
  return launched();
}

ewh_status ewh_f32_to_bf16(const float* a, void* b, long long n, void* stream) {
  if (!a || !b || n < 0) return nfail("ewh_f32_to_bf16: bad arguments");
  f32_to_bf16_kernel<<<egrid(n), 256, 0, (cudaStream_t)stream>>>(a, (bf16*)b, n);
  return launched();
}

ewh_status ewh_scaled_l2_loss(const float* y, const float* t, float* grad, float* loss, long long P, int C, int Cu,
                              int N, void* stream) {
  if (!y || !t || !grad || !loss || P < 1 || Cu < 1 || Cu > C || N < 1) return nfail("ewh_scaled_l2_loss: bad arguments");
  scaled_l2_kernel<<<N, 256, 0, (cudaStream_t)stream>>>(y, t, grad, loss, P, C, Cu, N);
  return launched();
}

ewh_status ewh_adam_step(float* param, const float* grad, float* m, float* v, void* param_bf16, long long n, float lr,
                         float beta1, float beta2, float eps, int step, void* stream) {
  if (!param || !grad || !m || !v || n < 0 || step < 1) return nfail("ewh_adam_step: bad arguments");
  const float c1 = 1.f - powf(beta1, (float)step), c2 = 1.f - powf(beta2, (float)step);
  adam_kernel<<<egrid(n), 256, 0, (cudaStream_t)stream>>>(param, grad, m, v, (bf16*)param_bf16, n, lr, beta1, beta2,
                                                          eps, c1, c2);
  return launched();
}

}  // extern "C"
