// Float-float arithmetic of the weight fit: a value as an unevaluated sum of two FP32
// numbers (this GPU's FP64 pipe is narrow).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace pmd {

// A double as a float-float pair (hi + lo within 2^-47 of x) with integer operations
// when its exponent is in [-70, 120] (this GPU's FP64 pipe is narrow; timings,
// predictions and residuals are well inside that range), else by FP64 conversions.
__device__ __forceinline__ float2 ff_of_double(double x) {
  const uint64_t b = (uint64_t)__double_as_longlong(x);
  const int e = (int)((b >> 52) & 0x7FF) - 1023;
  if (e < -70 || e > 120) {
    const float h = __double2float_rn(x);
    return make_float2(h, __double2float_rn(x - (double)h));
  }
  const uint32_t sgn = (uint32_t)(b >> 32) & 0x80000000u;
  const uint64_t m = b & 0xFFFFFFFFFFFFFull;                      // 52 fraction bits
  // hi: the leading one and the next 23 bits (truncated); lo: the 29 bits below, rounded
  const float h = __uint_as_float(sgn | ((uint32_t)(e + 127) << 23) | (uint32_t)(m >> 29));
  const float l = __uint2float_rn((uint32_t)(m & 0x1FFFFFFFu)) * __uint_as_float((uint32_t)(e - 52 + 127) << 23);
  return make_float2(h, sgn ? -l : l);
}

// float-float helpers: error-free product by FMA, compensated accumulation
__device__ __forceinline__ float2 ff_mul(float ah, float al, float bh, float bl) {
  const float p = __fmul_rn(ah, bh);
  float e = __fmaf_rn(ah, bh, -p);
  e = __fmaf_rn(ah, bl, e);
  e = __fmaf_rn(al, bh, e);
  return make_float2(p, e);
}
__device__ __forceinline__ void ff_acc(float &s, float &c, float2 p) {
  const float t = __fadd_rn(s, p.x);
  const float z = __fsub_rn(t, s);
  c = __fadd_rn(c, __fadd_rn(__fadd_rn(__fsub_rn(s, __fsub_rn(t, z)), __fsub_rn(p.x, z)), p.y));
  s = t;
}

// The same with the sum's own rounding errors kept: s + c + d holds the exact sum to some 2^-66
// of the largest part, so one FP64 sum of the three is no worse than adding in FP64.
__device__ __forceinline__ void two_sum(float &s, float x, float &err) {   // s + x = (new s) + err
  const float t = __fadd_rn(s, x), z = __fsub_rn(t, s);
  err = __fadd_rn(__fsub_rn(s, __fsub_rn(t, z)), __fsub_rn(x, z));
  s = t;
}
__device__ __forceinline__ void ff_acc3(float &s, float &c, float &d, float2 p) {
  float e0, e1, e2, e3;
  two_sum(p.x, p.y, e0);   // the leading bits in the first part, also where sums cancelled
  two_sum(s, p.x, e1);
  two_sum(c, e1, e2);
  two_sum(c, e0, e3);
  d = __fadd_rn(d, __fadd_rn(e2, e3));
}

}  // namespace pmd
