// FP64 reciprocal and reciprocal square root for serial chains.  An FP64 instruction takes 64 clocks
// here, the library's division 650 and its square root 670.
#pragma once
#include <cuda_runtime.h>

namespace dfscf {

// Householder's iterations of third order from an FP32 seed of the mantissa (A. S. Householder,
// The Numerical Treatment of a Single Nonlinear Equation, 1970): y (1 + e/2 + 3 e^2/8) with e =
// 1 - m y^2 for the square root, y (1 + e + e^2) with e = 1 - m y for the reciprocal.  5 and 3 FP64
// instructions instead of about 10 for the library's square root and division, to 2 ulp.  Arguments
// of ordinary size only.  Compared with 1 / sqrt(a) and 1 / a in tests/test_gpu_fp64_roots.py.
__device__ __forceinline__ bool ordinary(double a) {
  const int ex = (__double2hiint(a) >> 20) & 0x7ff;
  return ex > 200 && ex < 1846;
}
__device__ __forceinline__ float mantissa_f(int hi, int lo, int exponent) {
  return __int_as_float(((exponent) << 23) | ((hi & 0xfffff) << 3) | ((unsigned)lo >> 29));
}
__device__ __forceinline__ double widen(float f) {
  const int b = __float_as_int(f);
  return __hiloint2double((b >> 3) + 0x38000000, b << 29);
}
__device__ __forceinline__ double rsqrt_ordinary(double a) {
  const int hi = __double2hiint(a), lo = __double2loint(a);
  const int ex = (hi >> 20) - 1023, odd = ex & 1, half = (ex - odd) / 2;
  const double m = __hiloint2double((hi & 0xfffff) | ((1023 + odd) << 20), lo);  // in [1, 4)
  const double r = widen(rsqrtf(mantissa_f(hi, lo, 127 + odd)));
  const double er = fma(-(m * r), r, 1.0);
  const double q = fma(r * er, fma(0.375, er, 0.5), r);
  return __hiloint2double(__double2hiint(q) - (half << 20), __double2loint(q));
}
__device__ __forceinline__ double rcp_ordinary(double a) {
  const int hi = __double2hiint(a), lo = __double2loint(a);
  const int ex = ((hi >> 20) & 0x7ff) - 1023;
  const double m = __hiloint2double((hi & 0xfffff) | (1023 << 20), lo);  // in [1, 2)
  float seed;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(seed) : "f"(mantissa_f(hi, lo, 127)));
  const double r = widen(seed);
  const double er = fma(-m, r, 1.0);
  const double q = fma(r, fma(er, er, er), r);
  return __hiloint2double(__double2hiint(q) - (ex << 20), __double2loint(q));
}

}  // namespace dfscf
