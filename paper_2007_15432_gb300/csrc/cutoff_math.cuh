// Arithmetic of the cut-off radii, shared by the context's kernels (tree.cu) and
// the allocation-free ones (noalloc.cu).
#pragma once

#include "p3t_internal.cuh"

// 1 / sqrt(x) and x^(-1/4) from the 20-bit seed y by the binomial series (one
// rounding more than the last at most; the seed's range and bound are
// rsqrt_seed's, otherwise out of line): y (1 + e / 2 + 3/8 e^2) with e = 1 - x y^2;
// z (1 + e / 4 + 5/32 e^2 + 15/128 e^3) with z = y times the seed of y^(-1/2) and
// e = 1 - x z^4 (|e| < 2^-17), the rest below 2^-71.  5 and 8 FP64 instructions.
// rsqrt() for inv_sqrt: the radii of 1e6 bodies 205 -> 209 us.
__device__ __forceinline__ bool seed_range(double x) {
  return (unsigned)((__double2hiint(x) >> 20) - 512) < 1024u;
}
__device__ __forceinline__ double rsqrt_raw(double x) {
  double y;
  asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
  return y;
}
__device__ __forceinline__ double inv_sqrt(double x) {  // 0 for 0
  const double y = rsqrt_raw(x), e = __fma_rn(-x, y * y, 1.0);
  double r = __fma_rn(y * e, __fma_rn(e, 0.375, 0.5), y);
  if (!seed_range(x)) r = rsqrt_rare(x);
  return r;
}
static __device__ __noinline__ double inv_root4_rare(double x) { return rsqrt(sqrt(x)); }
__device__ __forceinline__ double inv_root4(double x) {
  const double y = rsqrt_raw(x), z = y * rsqrt_raw(y), z2 = z * z;
  const double e = __fma_rn(-x, z2 * z2, 1.0);
  double r = __fma_rn(z * e, __fma_rn(e, __fma_rn(e, 15.0 / 128.0, 5.0 / 32.0), 0.25), z);
  if (!seed_range(x)) r = inv_root4_rare(x);
  return r;
}

// x > 0 cut to FP32's 24 bits; within 2^+-100
__device__ __forceinline__ float cut_float(double x) {
  return __uint_as_float((unsigned)(__double2hiint(x) - (896 << 20)) << 3 |
                         (unsigned)__double2loint(x) >> 29);
}
__device__ __forceinline__ bool cut_range100(double x) {
  return (unsigned)((__double2hiint(x) >> 20) - (1023 - 100)) < 200u;
}
// (1 / Rmin^2, nb / (lmax - lmin)); zeros (no estimate) out of range
__device__ __forceinline__ float2 cut_scale(double Rmin, double lmin, double lmax, int nb) {
  const double q = Rmin * Rmin, span = lmax - lmin;
  if (!cut_range100(q) || !cut_range100(span)) return make_float2(0.f, 0.f);
  return make_float2(1.0f / cut_float(q), (float)nb / (float)span);
}
// bin of ln R among nb bins uniform on [lmin, lmax]: floor(nb (ln R - lmin) /
// (lmax - lmin)) clamped to [0, nb - 1], decided in FP64.  An FP32 estimate
// nb / (2 span) ln(R^2 / Rmin^2) decides it first when no integer lies within
// its error bound of the estimate: the squares cut to 24 bits, their quotient's
// two roundings and logf's last place leave the logarithm within 3.6e-7 + 1.2e-7
// of itself (2.4e-7 of the scale after the half), the scale's and the products'
// roundings are 3e-7 relative; the bound is 1.7 times the one and 3.3 times the
// other.  (One particle in a thousand is left at 377 bins over a
// factor e; a bound ten times wider sent a warp in four through the FP64
// logarithm.)  Otherwise the FP64 expression is evaluated.
static __device__ __noinline__ int cut_bin_fp64(double R2, double Rmin, double Rmax, double lmin,
                                                double lmax, int nb) {
  const double R = sqrt(R2);
  if (!(Rmax > Rmin && R > Rmin)) return 0;
  const double f = floor((log(R) - lmin) / (lmax - lmin) * (double)nb);
  // a NaN (a particle on the axis: lmin is -infinity) takes bin 0; its conversion
  // to int would be the smallest one
  return !(f >= 0.0) ? 0 : (f > (double)(nb - 1) ? nb - 1 : (int)f);
}
__device__ __forceinline__ int cut_bin(double R2, float2 sc, double Rmin, double Rmax, double lmin,
                                       double lmax, int nb) {
  const float tf = 0.5f * logf(cut_float(R2) * sc.x) * sc.y;
  const float margin = 4e-7f * sc.y + 1e-6f * (float)nb;
  const float lo = floorf(tf - margin);
  if (cut_range100(R2) && sc.y > 0.0f && margin < 0.25f && tf > -1.0f &&
      tf < 1.25f * (float)nb + 1.0f && lo == floorf(tf + margin))
    return min(max((int)lo, 0), nb - 1);
  return cut_bin_fp64(R2, Rmin, Rmax, lmin, lmax, nb);
}

// x^(1/3) for x >= 0: the inverse cube root z = x^(-1/3) from an FP32 seed
// (relative error below 5e-7), corrected once by the binomial series: with e = 1 -
// x z^3, z (1 + e / 3 + 2/9 e^2), the rest below 2^-60; then x^(1/3) = x z^2.  Inputs outside the
// seed's range take cbrt.  Conversions by integer operations (an FP64 one
// takes the FP64 pipe).
static __device__ __noinline__ double cbrt_rare(double x) { return cbrt(x); }
__device__ __forceinline__ double cbrt_pos(double x) {
  const unsigned f = __float_as_uint(rcbrtf(lead_float(x, 0)));
  const double z = __hiloint2double((int)((f >> 3) + (896u << 20)), (int)(f << 29));
  const double e = __fma_rn(-x, z * z * z, 1.0);
  const double w = __fma_rn(z * e, __fma_rn(e, 2.0 / 9.0, 1.0 / 3.0), z);
  double r = x * w * w;
  if ((unsigned)((__double2hiint(x) >> 20) - (1023 - 99)) >= 198u) r = cbrt_rare(x);
  return r;
}
