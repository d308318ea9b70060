// Helpers shared by the all-pairs sweeps: Blackwell's packed f32x2
// arithmetic (two FP32 values in one 64-bit register pair, one instruction),
// the MUFU reciprocal square root, TwoSum accumulation, the status poll, and
// the FP64 inverse cube distance.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "bd_internal.h"

namespace bdf {

typedef unsigned long long u64;

__device__ __forceinline__ float rsqrt_apx(float x) {
  float y;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// hi + lo += t with the rounding error of the high part kept in lo
__device__ __forceinline__ void two_sum(float &hi, float &lo, float t) {
  float s = __fadd_rn(hi, t);
  float bp = __fsub_rn(s, hi);
  float err = __fadd_rn(__fsub_rn(hi, __fsub_rn(s, bp)), __fsub_rn(t, bp));
  hi = s;
  lo = __fadd_rn(lo, err);
}

__device__ __forceinline__ int ctl_failed(const BdCtl *ctl) { return *(volatile const int *)&ctl->status; }

__device__ __forceinline__ u64 pk2(float a, float b) {
  u64 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ void up2(u64 r, float &a, float &b) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(r));
}
__device__ __forceinline__ u64 fma2(u64 a, u64 b, u64 c) {
  u64 d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ u64 sub2(u64 a, u64 b) {
  u64 d;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ u64 add2(u64 a, u64 b) {
  u64 d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ u64 mul2(u64 a, u64 b) {
  u64 d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
// the rounded sums of two packed pairs, and their rounding errors
__device__ __forceinline__ u64 two_sum2(u64 a, u64 b, u64 &err) {
  const u64 s = add2(a, b);
  const u64 bp = sub2(s, a);
  err = add2(sub2(a, sub2(s, bp)), sub2(b, bp));
  return s;
}

// x^(-3/2) for finite x > 0, in six FP64 instructions (FP64 issues at 1/64 of
// the FP32 rate on this part).  x = m 2^(2k), m in [1, 4); y = rsqrt(m) 2^-k to
// about 2^-22 from the FP32 unit, its bits moved between the formats by
// integer operations; then one step of (1 - e)^(-3/2) = 1 + 3/2 e + 15/8 e^2 +
// ..., e = 1 - x y^2, whose next term is below 2^-63.  (x = 0 gives inf, as a
// division would.)
__device__ __forceinline__ double inv_r3(double x) {
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
  const int k = ((int)(hi >> 20) - 1023) >> 1;
  const unsigned k20 = (unsigned)k * (1u << 20);
  // m truncated to FP32: bias 1023 -> 127, 20 + 3 mantissa bits
  const unsigned mb = ((hi - 2u * k20 - (896u << 20)) << 3) | (lo >> 29);
  const unsigned yb = __float_as_uint(rsqrt_apx(__uint_as_float(mb)));   // in (0.5, 1]
  const double y = __hiloint2double((int)((yb >> 3) + (896u << 20) - k20), (int)(yb << 29));
  const double y2 = __dmul_rn(y, y);   // exact: 24 x 24 bits
  const double e = __fma_rn(-x, y2, 1.0);
  const double y3 = __dmul_rn(y2, y);
  return __fma_rn(__dmul_rn(e, y3), __fma_rn(e, 1.875, 1.5), y3);
}

// |v| > h for v not NaN and h >= 0, by their bits (no FP64 compare)
__device__ __forceinline__ bool abs_above(double v, double h) {
  return (__double_as_longlong(v) & 0x7FFFFFFFFFFFFFFFll) > __double_as_longlong(h);
}

}  // namespace bdf
