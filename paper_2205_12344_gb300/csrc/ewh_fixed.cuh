// Block fixed point: sums and products of FP64 values on the integer pipe.
//
// One FP64 instruction of a GB300 SM takes the issue time of some forty 32-bit
// integer ones (2 lanes against 64 per clock), and two thirds of a leapfrog
// level's FP64 instructions are the differences 12 D, whose weights are the
// integers 1, 8.  The step kernels therefore quantise a tile's operands to 64-bit
// integers that share the tile's largest exponent, difference and multiply
// them exactly or with one truncation, and return to FP64 for the update.
//
// Accuracy: an operand keeps 56 or 57 bits below the tile's largest magnitude
// (FP64 keeps 53 below its own), the differences are exact, and a product keeps
// the upper 64 of 128 bits.  The acceleration's error stays below the
// rounding of the update u + delta that follows it (figures at the kernels).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace ewh {

using i64 = long long;

// Largest ratio (as a power of two) between a tile's largest modulus and its
// smallest mu that the fixed-point steps take: beyond it the rounding of a soft
// node's stresses, 2^-56 of the stiffest one's, would pass that of u + delta.
constexpr int FX_CONTRAST = 6;

// FP64 bits: sign-free upper word (exponent and leading mantissa bits)
__host__ __device__ __forceinline__ unsigned fx_key(double v) {
#ifdef __CUDA_ARCH__
  return (unsigned)__double2hiint(v) & 0x7fffffffu;
#else
  union { double d; uint64_t u; } c;
  c.d = v;
  return (unsigned)(c.u >> 32) & 0x7fffffffu;
#endif
}

// v 2^(BITS - (E - 1022)) as an integer; E the biased exponent of the largest
// magnitude (so the result is at most 2^BITS).  53 <= BITS <= 61.  ROUND: to the
// nearest (else towards zero).  Zero and denormal v give 0.
template <int BITS, bool ROUND>
__host__ __device__ __forceinline__ i64 fx_from(double v, int E) {
#ifdef __CUDA_ARCH__
  const unsigned hi = (unsigned)__double2hiint(v), lo = (unsigned)__double2loint(v);
#else
  union { double d; uint64_t u; } c;
  c.d = v;
  const unsigned hi = (unsigned)(c.u >> 32), lo = (unsigned)c.u;
#endif
  const int e = (int)((hi >> 20) & 0x7ffu);
  const uint64_t m = ((uint64_t)((hi & 0xfffffu) | 0x100000u) << 32) | lo;
  int s = E - e;
  if (s > 63 || e == 0) s = 63;
  const i64 q = ROUND ? (i64)(((m << (BITS - 52)) >> s) + 1) >> 1 : (i64)((m << (BITS - 53)) >> s);
  return (int)hi < 0 ? -q : q;
}

// A value as two signed 32-bit digits, v = hi 2^32 + lo.
struct FxSplit {
  int hi, lo;
};
__host__ __device__ __forceinline__ FxSplit fx_split(i64 v) {
  FxSplit r;
  r.lo = (int)v;
  r.hi = (int)(v >> 32) - (r.lo >> 31);
  return r;
}
// a b 2^-64 from three 32-bit products, the middle ones rounded; the product of
// the low digits (at most a quarter of a unit, of either sign) is dropped.
// |hi| <= 2^30 of at least one factor, so that the middle sum fits.
__host__ __device__ __forceinline__ i64 fx_mulhi(FxSplit a, FxSplit b) {
  i64 m = (i64)a.hi * b.lo + 0x80000000ll;
  m += (i64)a.lo * b.hi;
  return (i64)a.hi * b.hi + (m >> 32);
}

// 12 times the interior row of the first derivative, exact
__host__ __device__ __forceinline__ i64 fx_c12(i64 m2, i64 m1, i64 p1, i64 p2) { return (m2 - p2) + ((p1 - m1) << 3); }

// Taps of 12 D at a line position of class c (0 .. 3: closure rows of the low
// side, 4: interior, 5 .. 8: of the high side): offsets and weights scaled by
// 2^FX_TAP.  Every |weight| is below 32.
constexpr int FX_TAP = 57;
struct FxTaps {
  int off[4 * 9];
  i64 w[4 * 9];
};

// sum of weight x value over four taps, rounded, 2^-FX_TAP taken out
__host__ __device__ __forceinline__ i64 fx_taps(const i64* w, i64 a, i64 b, i64 c, i64 d) {
  __int128 s = (__int128)w[0] * a + (__int128)w[1] * b + (__int128)w[2] * c + (__int128)w[3] * d;
  return (i64)((s + ((i64)1 << (FX_TAP - 1))) >> FX_TAP);
}

// one weight x value, rounded
__host__ __device__ __forceinline__ i64 fx_taps_one(i64 w, i64 a) {
  return (i64)(((__int128)w * a + ((i64)1 << (FX_TAP - 1))) >> FX_TAP);
}

// 2^x as FP64 (-1022 <= x <= 1023)
__host__ __device__ __forceinline__ double fx_pow2(int x) {
#ifdef __CUDA_ARCH__
  return __hiloint2double((x + 1023) << 20, 0);
#else
  union { double d; uint64_t u; } c;
  c.u = (uint64_t)(x + 1023) << 52;
  return c.d;
#endif
}

}  // namespace ewh
