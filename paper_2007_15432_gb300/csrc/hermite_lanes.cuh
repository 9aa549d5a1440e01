// Pieces shared by the kernels that integrate small clusters with their members
// spread over the lanes of a warp (the forward block steps of hard.cu, the
// tangents of hermite_adj.cu).
#pragma once

#include <math.h>

#include "p3t_internal.cuh"

// what the block steps take from (dt, parameters), formed once on the host in
// the same IEEE operations
struct HConst {
  double unit, unit6;       // dt / 2^40, 6 unit
  double m52u;              // -2^52 unit
  double c3u, c4u, c5u;     // unit^3 / 6, unit^4 / 24, unit^5 / 120
  double idt2, idt3;        // 1 / dt^2, 1 / dt^3
  double i1mg, gms;         // 1 / (1 - gamma), G M_*
  float etaf, eta0f;
  float gin2;               // (y r_out)^2 below this in FP32: y < gamma in FP64
  int fast;                 // the constants stay normal at every level
};

// a step of level l is D = unit 2^(40 - l) exactly, so D^n = RN(unit^n)
// 2^(n (40 - l)) and RN(D^n c) = RN(unit^n c) 2^(n (40 - l)) with unit^n
// formed by successive products: the corrector's powers of D and of 1/D are
// these constants shifted in the exponent (the same bits as the products, no
// FP64 instruction)
static inline HConst hermite_const(const p3t_params &prm, double dt) {
  HConst h;
  h.unit = ldexp(dt, -P3T_KMAX);
  h.unit6 = 6.0 * h.unit;
  h.m52u = -4503599627370496.0 * h.unit;
  const double u2 = h.unit * h.unit, u3 = u2 * h.unit, u4 = u3 * h.unit, u5 = u4 * h.unit;
  h.c3u = u3 * (1.0 / 6.0);
  h.c4u = u4 * (1.0 / 24.0);
  h.c5u = u5 * (1.0 / 120.0);
  const double idt = 1.0 / dt;
  h.idt2 = idt * idt;
  h.idt3 = h.idt2 * idt;
  h.i1mg = 1.0 / (1.0 - prm.gamma);
  h.gms = prm.G * prm.m_star;
  h.etaf = (float)prm.eta;
  h.eta0f = (float)prm.eta0;
  h.gin2 = (float)(prm.gamma * prm.gamma * (1.0 - 1e-5));
  h.fast = dt >= 1e-30 && dt <= 1e30;
  return h;
}

__device__ __forceinline__ double shfl_d(double v, int src) {
  return __shfl_sync(0xffffffffu, v, src);
}
// a > b and a >= b for a >= 0 or NaN and b >= 0 from the bit patterns (an FP64
// comparison takes an FP64 slot); false for NaN
__device__ __forceinline__ bool gt_pos(double a, double b) {
  const long long x = __double_as_longlong(a);
  return x > __double_as_longlong(b) && x <= 0x7ff0000000000000LL;
}
__device__ __forceinline__ bool ge_pos(double a, double b) {
  const long long x = __double_as_longlong(a);
  return x >= __double_as_longlong(b) && x <= 0x7ff0000000000000LL;
}
// x 2^k for x and x 2^k normal
__device__ __forceinline__ double shift_exp(double x, int k) {
  return __hiloint2double(__double2hiint(x) + (k << 20), __double2loint(x));
}
// minimum over the warp of a value in [0, 2^63): the minimum of the high
// words, then of the low words among the lanes that hold it (two warp
// reductions instead of five dependent shuffle steps)
__device__ __forceinline__ int64_t warp_min64(int64_t v) {
  const unsigned hi = (unsigned)((unsigned long long)v >> 32), lo = (unsigned)v;
  const unsigned hmin = __reduce_min_sync(0xffffffffu, hi);
  const unsigned lmin = __reduce_min_sync(0xffffffffu, hi == hmin ? lo : 0xffffffffu);
  return (int64_t)(((unsigned long long)hmin << 32) | lmin);
}

// quantise_level for a normal positive dt (with every dt / 2^k normal), from
// the bit patterns: dt / 2^l <= dt_des iff bits(dt) - (l << 52) <= bits(dt_des)
__device__ __forceinline__ int level_bits(double dt_des, long long bd, int prev, int64_t t,
                                          bool &underflow) {
  const long long bs = __double_as_longlong(dt_des);
  int lvl = 0;
  if (bs < bd && (bs & 0x7fffffffffffffffLL) <= 0x7ff0000000000000LL) {
    const long long l = bs > 0 ? (bd - bs + 0xfffffffffffffLL) >> 52 : P3T_KMAX + 1;
    underflow = underflow || l > P3T_KMAX;
    lvl = l > P3T_KMAX ? P3T_KMAX : (int)l;
  }
  lvl = max(lvl, prev - 1);
  if (t != 0) lvl = max(lvl, P3T_KMAX - __ffsll((long long)t) + 1);
  return min(lvl, P3T_KMAX);
}

// sum of the squares held by the three lanes from l0 on
__device__ __forceinline__ float norm_lanes(float x, int l0) {
  const float s = x * x;
  return __shfl_sync(0xffffffffu, s, l0 & 31) + __shfl_sync(0xffffffffu, s, (l0 + 1) & 31) +
         __shfl_sync(0xffffffffu, s, (l0 + 2) & 31);
}
__device__ __forceinline__ float sqrt_approx(float x) {
  float r;
  asm("sqrt.approx.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}

// The step criterion (the first step eta0 |a| / |j|, or, `later`, sqrt(eta (|a|
// |a2| + |j|^2) / (|j| |a3| + |a2|^2))) from squared norms good to 2e-6, by
// approximate roots and quotient: dtd = its value times 2^e, good to 1e-5.
// Returns whether dtd decides the level: it lies 2^-14 or more from every power
// of two times dt (bd: dt's bits), and every squared norm, product, sum and
// quotient formed is a normal number.  (The products of two squared norms are
// the first to leave FP32's range: accelerations of 1e-9 with steps of a
// twentieth of |a| / |j| have |j|^2 |a3|^2 of 4e-47.)
__device__ __forceinline__ bool step_estimate(float an, float jn, float a2n, float a3n, int e,
                                              bool later, const HConst &hc, long long bd,
                                              double &dtd) {
  float r;
  bool fine = an > 1e-30f && an < 1e30f && jn > 1e-30f && jn < 1e30f;
  if (later) {
    const float p = an * a2n, q = jn * a3n;
    const float num = hc.etaf * (sqrt_approx(p) + jn), den = sqrt_approx(q) + a2n;
    const float s = __fdividef(num, den);
    r = sqrt_approx(s);
    fine = fine && a2n > 1e-30f && a2n < 1e30f && a3n > 1e-30f && a3n < 1e30f && p > 1e-37f &&
           q > 1e-37f && num > 1e-37f && s > 1e-37f;
  } else {
    const float s = __fdividef(an, jn);
    r = hc.eta0f * sqrt_approx(s);
    fine = fine && s > 1e-37f;
  }
  const unsigned u = __float_as_uint(r);
  const int er = (int)(u >> 23) - 127 + 1023 + e;
  fine = fine && r > 1e-30f && r < 1e30f && er > 0 && er < 2047;
  const long long bs = (long long)er << 52 | (long long)(u & 0x7fffffu) << 29;
  const long long frac = (bs - bd) & 0xfffffffffffffLL, lim = 1LL << 38;
  dtd = __longlong_as_double(bs);
  return fine && frac >= lim && frac <= (1LL << 52) - lim;
}
