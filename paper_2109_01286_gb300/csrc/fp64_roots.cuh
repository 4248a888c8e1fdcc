// FP64 reciprocal and reciprocal square root from an FP32 seed.
//
// GB300 runs one FP64 warp instruction per SM in 16 clocks, as long as 64 integer or FP32 lane
// operations per lane, so the iterations take as few FP64 operations as the seed allows: with
// y0 = x^(-1/2) (1 + d) and e = 1 - x y0^2, x^(-1/2) = y0 (1 - e)^(-1/2) = y0 (1 + e/2 + 3 e^2/8 +
// O(e^3)) (the binomial series, Householder's third-order step), and 1/x = r0 (1 + e + e^2 + O(e^3))
// with e = 1 - x r0.  The seed (FP32 hardware rsqrt / reciprocal of x truncated to 24 bits) leaves
// |e| < 2^-20, so the series' remainders are below 2^-60.  Five and three FP64 operations; largest
// error over 2^22 arguments against long double roots and quotients: 0.991 and 0.500 ulp (positive normal
// arguments; others go to the CUDA functions).
#pragma once
#include <cuda_runtime.h>

namespace hfd {

// Bits of the positive normal FP64 value (hi, lo), of exponent in the float range, as a truncated
// float, and a positive normal float widened.
__device__ __forceinline__ float seed_f32(int hi, int lo) {
  return __int_as_float(((hi - (896 << 20)) << 3) | (int)((unsigned)lo >> 29));
}
__device__ __forceinline__ double seed_f64(float f, int exp_add) {
  const int b = __float_as_int(f);
  return __hiloint2double((b >> 3) + (896 << 20) + (exp_add << 20), b << 29);
}
__device__ __forceinline__ bool positive_normal(double x) {
  return (unsigned)__double2hiint(x) - 0x00100000u < 0x7fe00000u;
}

__device__ __forceinline__ double rsqrt64(double x) {
  if (!positive_normal(x)) return rsqrt(x);
  const int hi = __double2hiint(x);
  const int k = ((hi >> 20) - 1023) & ~1;                       // x = m 2^k, 1 <= m < 4
  const float m = seed_f32(hi - (k << 20), __double2loint(x));
  const double y = seed_f64(rsqrtf(m), -(k >> 1));
  const double e = __fma_rn(-__dmul_rn(x, y), y, 1.0);
  return __fma_rn(__dmul_rn(y, e), __fma_rn(0.375, e, 0.5), y);
}

__device__ __forceinline__ double rcp64(double x) {
  if (!positive_normal(x)) return 1.0 / x;
  const int hi = __double2hiint(x);
  const int k = (hi >> 20) - 1023;                              // x = m 2^k, 1 <= m < 2
  if (k > 1000) return 1.0 / x;                                 // the result may be subnormal
  const float m = seed_f32(hi - (k << 20), __double2loint(x));
  const double r = seed_f64(__fdividef(1.0f, m), -k);
  const double e = __fma_rn(-x, r, 1.0);
  return __fma_rn(r, __fma_rn(e, e, e), r);
}

// x > 0 (false for NaN; infinity passes), on the integer pipe.
__device__ __forceinline__ bool positive_bits(double x) {
  const int hi = __double2hiint(x);
  return hi >= 0 && (hi | __double2loint(x)) != 0 &&
         ((unsigned)hi < 0x7ff00000u || ((unsigned)hi == 0x7ff00000u && __double2loint(x) == 0));
}

}  // namespace hfd
