// Order-zero Boys function F0(t) = int_0^1 exp(-t u^2) du on the GPU.
//
// Every s-type Coulomb integral of the density-fitting path ((P|Q), (Q|mn), and the
// nuclear attraction) reduces to a prefactor times F0 of a scaled squared distance.
// One lane evaluates one integral; the three regimes below are chosen per lane and the
// far regime (most pairs of a large molecule) needs only one square root and division.
//   t < 1e-3 : Maclaurin series sum_k (-t)^k / (k! (2k+1)), seven terms (truncation
//              error below 1e-22);
//   t > 40   : erf(sqrt t) equals 1 in double precision, F0 = (sqrt(pi)/2) / sqrt(t);
//   otherwise: F0 = (sqrt(pi)/2) erf(sqrt t) / sqrt t, with CUDA's erf.
#pragma once

__device__ __forceinline__ double boys_f0(double t) {
  const double half_sqrt_pi = 0.88622692545275801365;
  if (t < 1e-3) {
    // coefficients 1/(k! (2k+1)) with alternating signs, Horner in t
    double r = 1.0 / 9360.0;
    r = fma(r, -t, 1.0 / 1320.0);
    r = fma(r, -t, 1.0 / 216.0);
    r = fma(r, -t, 1.0 / 42.0);
    r = fma(r, -t, 1.0 / 10.0);
    r = fma(r, -t, 1.0 / 3.0);
    return fma(r, -t, 1.0);
  }
  double s = sqrt(t);
  if (t > 40.0) return half_sqrt_pi / s;
  return half_sqrt_pi * erf(s) / s;
}

// ---- tabulated F0 ------------------------------------------------------------------------
// FP64 issues at 2 lanes/clk/SM here, and erf, the square roots and the divisions of one Coulomb
// integral take about 140 FP64 instructions.  The integral kernels below 40 therefore use the
// Taylor series F0(t0 + d) = sum_j (-d)^j F_j(t0) / j! around the nearest t0 = k / 32 (degree 6:
// the remainder is under 2^-55 of F0), and one reciprocal square root above.  The table (1281
// rows of 8 doubles, 82 KB) stays in L1; a kernel fills it before the integrals, as
// it takes 3 us.
constexpr int BOYS_ROWS = 40 * 32 + 1, BOYS_STRIDE = 8;
constexpr size_t BOYS_TABLE = (size_t)BOYS_ROWS * BOYS_STRIDE;

// 1 / sqrt(a) to about 1 ulp in 5 FP64 instructions: the hardware's 2^-20 estimate and one step of
// third order (Householder): y (1 + e/2 + 3 e^2/8), e = 1 - a y^2 (tests/test_gpu_fp64_roots.py).
__device__ __forceinline__ double rsqrt_fast(double a) {
  const unsigned h = (unsigned)__double2hiint(a);
  if (h - 0x00100000u >= 0x7fd00000u) return 1.0 / sqrt(a);  // not a positive normal number below 2^1023
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(a));
  const double e = fma(-(a * y), y, 1.0);
  return fma(y * e, fma(0.375, e, 0.5), y);
}

__device__ __forceinline__ double boys_f0_table(double t, const double* __restrict__ table) {
  if ((unsigned)__double2hiint(t) >= 0x40440000u) {  // 40 and above, NaN
    return 0.88622692545275801365 * rsqrt_fast(t);
  }
  const double m = fma(t, 32.0, 6755399441055744.0);  // 1.5 2^52: rounds to an integer
  const double d = fma(m - 6755399441055744.0, -0.03125, t);
  const double2* c = reinterpret_cast<const double2*>(table + (size_t)__double2loint(m) * BOYS_STRIDE);
  const double2 c01 = __ldg(c), c23 = __ldg(c + 1), c45 = __ldg(c + 2);
  double r = __ldg(reinterpret_cast<const double*>(c + 3));
  r = fma(r, d, c45.y);
  r = fma(r, d, c45.x);
  r = fma(r, d, c23.y);
  r = fma(r, d, c23.x);
  r = fma(r, d, c01.y);
  return fma(r, d, c01.x);
}
