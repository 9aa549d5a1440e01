// Soft step: kick, Hermite-4 hard step of the neighbour
// clusters, Kepler drift of isolated particles, energy.
//
// Compiled with -fmad=false.  The Hermite force, predictor, corrector and
// step rule are evaluated in one fixed order with IEEE division and square
// root, so that the block-step schedule (decided by comparing FP64 step
// estimates with dt / 2^k) does not depend on the machine.
#include <type_traits>

#include "p3t_internal.cuh"
#include "exact_conv.cuh"
#include "hermite_lanes.cuh"

namespace {

constexpr int kBlock = 256;

// ---- soft kick (procedure steps 3 and 8) ------------------------------------
// Members of a composite formed by the last hard step (Sec. 2.4.1;
// slot[i] >= 0, its entry in ent) are kicked with the composite's mass-
// weighted mean acceleration sum_l m_l a_l / sum_l m_l (ascending l); the
// composite's lowest member records the dissipation sum_l m_l |h (a_l -
// a_c)|^2 / 2 at its entry.
__global__ void k_kick(int64_t n, double *vx, double *vy, double *vz,
                       const double *ax, const double *ay, const double *az,
                       double h, const int32_t *slot, const int4 *ent, const double *m,
                       double *esoft) {
  pdl_wait();
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    // every load before the first use of one (N = 1e6 20 -> 18 us, 1e4 4.8 -> 3.7)
    const int32_t s = slot ? slot[i] : -1;
    const double ux = vx[i], uy = vy[i], uz = vz[i], bx = ax[i], by = ay[i], bz = az[i];
    if (s < 0) {
      vx[i] = ux + bx * h;
      vy[i] = uy + by * h;
      vz[i] = uz + bz * h;
      continue;
    }
    const int4 e = ent[s];
    double M = 0.0, A[3] = {0.0, 0.0, 0.0};
    for (int l = e.z; l < e.w; ++l) {
      const int q = ent[l].x;
      M += m[q];
      A[0] += m[q] * ax[q]; A[1] += m[q] * ay[q]; A[2] += m[q] * az[q];
    }
    const double ac[3] = {A[0] / M, A[1] / M, A[2] / M};
    vx[i] = ux + ac[0] * h;
    vy[i] = uy + ac[1] * h;
    vz[i] = uz + ac[2] * h;
    if (e.x == e.y) {
      double Es = 0.0;
      for (int l = e.z; l < e.w; ++l) {
        const int q = ent[l].x;
        const double dx = (ax[q] - ac[0]) * h, dy = (ay[q] - ac[1]) * h, dz = (az[q] - ac[2]) * h;
        Es += 0.5 * m[q] * (dx * dx + dy * dy + dz * dz);
      }
      esoft[s] = Es;
    }
  }
}

// ---- Kepler drift, universal variables --------------------------------------
// Stumpff functions C(z) = sum (-z)^k / (2k+2)!, S(z) = sum (-z)^k / (2k+3)!,
// as nested series for |z| < 1 (4 terms below |z| = 1e-3, 6 below 1e-2, 10
// above; truncation below 1e-19 of the result in each band) and in closed
// form otherwise.
__device__ __forceinline__ void stumpff(double z, double &C, double &S) {
  constexpr double c0 = 1.0 / 2.0, c1 = -1.0 / 24.0, c2 = 1.0 / 720.0,
                   c3 = -1.0 / 40320.0, c4 = 1.0 / 3628800.0,
                   c5 = -1.0 / 479001600.0, c6 = 1.0 / 87178291200.0,
                   c7 = -1.0 / 20922789888000.0, c8 = 1.0 / 6402373705728000.0,
                   c9 = -1.0 / 2432902008176640000.0;
  constexpr double s0 = 1.0 / 6.0, s1 = -1.0 / 120.0, s2 = 1.0 / 5040.0,
                   s3 = -1.0 / 362880.0, s4 = 1.0 / 39916800.0,
                   s5 = -1.0 / 6227020800.0, s6 = 1.0 / 1307674368000.0,
                   s7 = -1.0 / 355687428096000.0, s8 = 1.0 / 121645100408832000.0,
                   s9 = -1.0 / 51090942171709440000.0;
  const double az = fabs(z);
  if (az < 1e-3) {
    double c = __fma_rn(z, c3, c2), s = __fma_rn(z, s3, s2);
    c = __fma_rn(z, c, c1); s = __fma_rn(z, s, s1);
    C = __fma_rn(z, c, c0); S = __fma_rn(z, s, s0);
  } else if (az < 1e-2) {
    double c = __fma_rn(z, c5, c4), s = __fma_rn(z, s5, s4);
    c = __fma_rn(z, c, c3); s = __fma_rn(z, s, s3);
    c = __fma_rn(z, c, c2); s = __fma_rn(z, s, s2);
    c = __fma_rn(z, c, c1); s = __fma_rn(z, s, s1);
    C = __fma_rn(z, c, c0); S = __fma_rn(z, s, s0);
  } else if (az < 1.0) {
    double c = __fma_rn(z, c9, c8), s = __fma_rn(z, s9, s8);
    c = __fma_rn(z, c, c7); s = __fma_rn(z, s, s7);
    c = __fma_rn(z, c, c6); s = __fma_rn(z, s, s6);
    c = __fma_rn(z, c, c5); s = __fma_rn(z, s, s5);
    c = __fma_rn(z, c, c4); s = __fma_rn(z, s, s4);
    c = __fma_rn(z, c, c3); s = __fma_rn(z, s, s3);
    c = __fma_rn(z, c, c2); s = __fma_rn(z, s, s2);
    c = __fma_rn(z, c, c1); s = __fma_rn(z, s, s1);
    C = __fma_rn(z, c, c0); S = __fma_rn(z, s, s0);
  } else if (z > 0.0) {
    const double q = sqrt(z);
    C = (1.0 - cos(q)) / z;
    S = (q - sin(q)) / (z * q);
  } else {
    const double q = sqrt(-z);
    C = (cosh(q) - 1.0) / (-z);
    S = (sinh(q) - q) / (-z * q);
  }
}

// Per-call constants of the drift: mu, sqrt(mu), 1 / sqrt(mu), 1 / mu.
struct KepConst {
  double mu, sq, isq, imu;
};

// Advances (X, V) by dt on the Kepler orbit about mu.  Universal anomaly chi
// solves F(chi) = sig chi^2 C + (1 - alpha r0) chi^3 S + r0 chi - sqrt(mu) dt
// = 0 (z = alpha chi^2, sig = r0 v_r0 / sqrt(mu)) by Newton-Raphson from the
// third-order series inversion of F; F'(chi) = r(chi) and F''(chi) = sig (1 -
// z C) + (1 - alpha r0) chi (1 - z S).  A Newton step d leaves an error of
// about |F'' / (2 F')| d^2, so the iteration stops once 16 times that bound
// is below 2^-53 |chi| (or |d| <= 1e-10 |chi|).  Then Lagrange f, g.
__device__ bool kepler_uv(double X[3], double V[3], double dt, const KepConst &K) {
  const double r02 = __fma_rn(X[0], X[0], __fma_rn(X[1], X[1], X[2] * X[2]));
  const double v2 = __fma_rn(V[0], V[0], __fma_rn(V[1], V[1], V[2] * V[2]));
  const double rv = __fma_rn(X[0], V[0], __fma_rn(X[1], V[1], X[2] * V[2]));
  const double ir0 = rsqrt(r02);
  const double r0 = r02 * ir0;
  const double alpha = __fma_rn(-v2, K.imu, 2.0 * ir0);
  const double sig = rv * K.isq;  // r0 v_r0 / sqrt(mu)
  const double tau = K.sq * dt;
  const double bet = __fma_rn(-alpha, r0, 1.0);
  // inversion of tau = r0 chi + sig chi^2 / 2 + bet chi^3 / 6 + O(chi^4)
  const double x1 = tau * ir0, hs = 0.5 * sig * ir0;
  double chi = x1 * __fma_rn(__fma_rn(hs, hs + hs, -bet * ir0 * (1.0 / 6.0) * ir0), x1 * x1,
                             __fma_rn(-hs, x1, 1.0));
  // beyond a quarter period (16 dt^2 alpha^3 mu > (2 pi)^2) start from the mean motion
  if (alpha > 0.0 && 16.0 * dt * dt * alpha * alpha * alpha * K.mu > 4.0 * 9.869604401089358)
    chi = tau * alpha;
  double C = 0.5, S = 1.0 / 6.0, z = 0.0;
  bool ok = false;
  for (int it = 0; it < 64; ++it) {
    z = alpha * chi * chi;
    stumpff(z, C, S);
    const double chi2 = chi * chi;
    const double F = __fma_rn(sig * chi2, C, __fma_rn(bet * chi2 * chi, S, __fma_rn(r0, chi, -tau)));
    const double Fp = __fma_rn(sig * chi, __fma_rn(-z, S, 1.0), __fma_rn(bet * chi2, C, r0));
    const double Fpp = __fma_rn(sig, __fma_rn(-z, C, 1.0), bet * chi * __fma_rn(-z, S, 1.0));
    const double iFp = 1.0 / Fp;
    double d = F * iFp;
    const double lim = 0.5 * (fabs(chi) + r0);
    if (d > lim) d = lim;
    if (d < -lim) d = -lim;
    chi -= d;
    const double rest = 0.5 * fabs(Fpp * iFp) * d * d;
    if (16.0 * rest <= 1.1102230246251565e-16 * fabs(chi) || fabs(d) <= 1e-10 * fabs(chi) ||
        d == 0.0) {
      ok = true;
      break;
    }
  }
  z = alpha * chi * chi;
  stumpff(z, C, S);
  const double chi2 = chi * chi;
  const double f = __fma_rn(-chi2 * ir0, C, 1.0);
  const double g = __fma_rn(-chi2 * chi, S * K.isq, dt);
  double nx[3];
  for (int a = 0; a < 3; ++a) nx[a] = __fma_rn(f, X[a], g * V[a]);
  const double ir = rsqrt(__fma_rn(nx[0], nx[0], __fma_rn(nx[1], nx[1], nx[2] * nx[2])));
  const double fd = K.sq * ir * ir0 * __fma_rn(z, S, -1.0) * chi;
  const double gd = __fma_rn(-chi2 * ir, C, 1.0);
  for (int a = 0; a < 3; ++a) {
    const double nv = __fma_rn(fd, X[a], gd * V[a]);
    X[a] = nx[a];
    V[a] = nv;
  }
  return ok;
}

__device__ __forceinline__ double ldexp_fast(double x, int k) {
  const long long b = __double_as_longlong(x);
  const int e = (int)((b >> 52) & 0x7ff);
  if (e > 0 && e < 0x7ff && e + k > 0 && e + k < 0x7ff)
    return __longlong_as_double(b + ((long long)k << 52));
  return ldexp(x, k);
}
__device__ __forceinline__ int ilogb_fast(double x) {
  const int e = (int)((__double_as_longlong(x) >> 52) & 0x7ff);
  return (e > 0 && e < 0x7ff) ? e - 1023 : ilogb(x);
}

// Conversions by integer operations.  On this part a conversion between FP64
// and FP32 or from an integer to FP64 takes the FP64 pipe like an FP64
// multiply (about 64 cycles of a sub-partition); along the serial block steps
// of a close encounter these sit on the critical path, so where the result is
// a normal number they are done on the bits instead, with the same results.
// (float)(a 2^k), rounded to nearest even, for a 2^k in FP32's normal range
// (the FP64 forms of the rare cases out of line: inlined, the compiler
// predicates them into every call, and predicated-off FP64 instructions still
// take the FP64 pipe)
__device__ __noinline__ float d2f_scaled_fp64(double a, int k) { return (float)ldexp_fast(a, k); }
__device__ __noinline__ double f2d_fp64(float f) { return (double)f; }
__device__ __noinline__ double i2d_fp64(int64_t x) { return (double)x; }
__device__ __forceinline__ float d2f_scaled(double a, int k) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(a);
  const int ed = (int)((b >> 52) & 0x7ff);
  const int ef = ed - 1023 + k + 127;
  if (ed == 0 || ed == 0x7ff || ef <= 0 || ef >= 255) return d2f_scaled_fp64(a, k);
  const unsigned long long m = b & 0xfffffffffffffull;
  unsigned r = ((unsigned)ef << 23) | (unsigned)(m >> 29);
  const unsigned long long rem = m & 0x1fffffffull, half = 0x10000000ull;
  if (rem > half || (rem == half && (r & 1u))) ++r;  // a carry into the exponent is right
  return __uint_as_float(r | ((unsigned)(b >> 32) & 0x80000000u));
}
// (double)f, exact
__device__ __forceinline__ double f2d_exact(float f) {
  const unsigned u = __float_as_uint(f);
  const int ef = (int)((u >> 23) & 0xff);
  if (ef == 0 || ef == 0xff) return f2d_fp64(f);
  return __longlong_as_double((long long)((unsigned long long)(u & 0x80000000u) << 32 |
                                          (unsigned long long)(ef - 127 + 1023) << 52 |
                                          (unsigned long long)(u & 0x7fffffu) << 29));
}
// (double)x for 0 <= x < 2^53, exact
__device__ __forceinline__ double i2d_exact(int64_t x) {
  if (x <= 0) return i2d_fp64(x);
  const int e = 63 - __clzll(x);
  return __longlong_as_double((long long)((unsigned long long)(e + 1023) << 52 |
                                          (((unsigned long long)x << (52 - e)) &
                                           0xfffffffffffffull)));
}

// Mixed path: the same drift in float-float arithmetic (FP32 instructions,
// ~2^-47 relative per operation) for bound orbits whose Stumpff argument
// stays below 1e-2 (a soft step is a small fraction of an orbit): the same
// universal-anomaly equation, the third-order start, Newton steps until the
// step is below 2^-44 of chi, Stumpff series to z^4 (the next term is below
// 1e-19 of the first), Lagrange f, g.  The FP64 pipe then carries only the
// splits of the state into float-float pairs and back.  Anything else (an
// unbound or long arc, no convergence in four steps) returns false and takes
// the FP64 solver, on the untouched state.  The drift's results agree with
// the FP64 solver's to ~1e-14 relative.
struct KepFF {
  FF sq, isq, imu;
};
// x = hi + lo with hi = (float)x and lo = (float)(x - hi) (the difference
// exact); the conversions on the bits, one FP64 subtraction
__device__ __forceinline__ FF ff_split(double x) {
  const float h = d2f_scaled(x, 0);
  return {h, d2f_scaled(x - f2d_exact(h), 0)};
}
__device__ __forceinline__ double ff_to_double(FF a) { return f2d_exact(a.h) + f2d_exact(a.l); }
__device__ __forceinline__ FF ff_sub(FF a, FF b) { return ff_add(a, ff_neg(b)); }
__device__ __forceinline__ FF ff_c(float h, float l) { return {h, l}; }
// the Stumpff series' coefficients as float-float constants
#define P3T_FFC(name, v) constexpr float name##h = (float)(v), name##l = (float)((v) - (double)(float)(v))
P3T_FFC(kC0, 1.0 / 2.0); P3T_FFC(kC1, -1.0 / 24.0); P3T_FFC(kC2, 1.0 / 720.0);
P3T_FFC(kC3, -1.0 / 40320.0); P3T_FFC(kC4, 1.0 / 3628800.0);
P3T_FFC(kS0, 1.0 / 6.0); P3T_FFC(kS1, -1.0 / 120.0); P3T_FFC(kS2, 1.0 / 5040.0);
P3T_FFC(kS3, -1.0 / 362880.0); P3T_FFC(kS4, 1.0 / 39916800.0);
#undef P3T_FFC
__device__ __forceinline__ void stumpff_ff(FF z, FF &C, FF &S) {
  FF c = ff_add(ff_c(kC3h, kC3l), ff_mul(z, ff_c(kC4h, kC4l)));
  FF t = ff_add(ff_c(kS3h, kS3l), ff_mul(z, ff_c(kS4h, kS4l)));
  c = ff_add(ff_c(kC2h, kC2l), ff_mul(z, c)); t = ff_add(ff_c(kS2h, kS2l), ff_mul(z, t));
  c = ff_add(ff_c(kC1h, kC1l), ff_mul(z, c)); t = ff_add(ff_c(kS1h, kS1l), ff_mul(z, t));
  C = ff_add(ff_c(kC0h, kC0l), ff_mul(z, c)); S = ff_add(ff_c(kS0h, kS0l), ff_mul(z, t));
}

__device__ bool kepler_ff(double X[3], double V[3], double dt, const KepFF &K) {
  const FF x[3] = {ff_split(X[0]), ff_split(X[1]), ff_split(X[2])};
  const FF v[3] = {ff_split(V[0]), ff_split(V[1]), ff_split(V[2])};
  const FF r02 = ff_add(ff_add(ff_mul(x[0], x[0]), ff_mul(x[1], x[1])), ff_mul(x[2], x[2]));
  const FF v2 = ff_add(ff_add(ff_mul(v[0], v[0]), ff_mul(v[1], v[1])), ff_mul(v[2], v[2]));
  const FF rv = ff_add(ff_add(ff_mul(x[0], v[0]), ff_mul(x[1], v[1])), ff_mul(x[2], v[2]));
  const FF ir0 = ff_rsqrt(r02);
  const FF r0 = ff_mul(r02, ir0);
  const FF alpha = ff_sub(ff_mulf(ir0, 2.0f), ff_mul(v2, K.imu));
  const FF sig = ff_mul(rv, K.isq);
  const FF dtf = ff_split(dt);
  const FF tau = ff_mul(K.sq, dtf);
  const FF bet = ff_sub(ff_c(1.0f, 0.0f), ff_mul(alpha, r0));
  // inversion of tau = r0 chi + sig chi^2 / 2 + bet chi^3 / 6 + O(chi^4)
  const FF x1 = ff_mul(tau, ir0), hs = ff_mulf(ff_mul(sig, ir0), 0.5f);
  const FF q = ff_sub(ff_mulf(ff_mul(hs, hs), 2.0f),
                      ff_mulf(ff_mul(ff_mul(bet, ir0), ir0), 1.0f / 6.0f));
  FF chi = ff_mul(x1, ff_add(ff_sub(ff_c(1.0f, 0.0f), ff_mul(hs, x1)),
                             ff_mul(q, ff_mul(x1, x1))));
  if (!(alpha.h > 0.0f)) return false;
  FF z = ff_mul(alpha, ff_mul(chi, chi)), C, S;
  bool conv = false;
  for (int it = 0; it < 4; ++it) {
    if (!(fabsf(z.h) < 1e-2f)) return false;
    stumpff_ff(z, C, S);
    const FF chi2 = ff_mul(chi, chi);
    const FF F = ff_sub(ff_add(ff_add(ff_mul(ff_mul(sig, chi2), C),
                                      ff_mul(ff_mul(bet, ff_mul(chi2, chi)), S)),
                               ff_mul(r0, chi)),
                        tau);
    const FF Fp = ff_add(ff_add(ff_mul(ff_mul(sig, chi), ff_sub(ff_c(1.0f, 0.0f), ff_mul(z, S))),
                                ff_mul(ff_mul(bet, chi2), C)),
                         r0);
    const FF d = ff_div(F, Fp);
    chi = ff_sub(chi, d);
    z = ff_mul(alpha, ff_mul(chi, chi));
    if (fabsf(d.h) <= 5.684341886080802e-14f * fabsf(chi.h)) {  // 2^-44
      conv = true;
      break;
    }
  }
  if (!conv || !(fabsf(z.h) < 1e-2f)) return false;
  stumpff_ff(z, C, S);
  const FF chi2 = ff_mul(chi, chi);
  const FF f = ff_sub(ff_c(1.0f, 0.0f), ff_mul(ff_mul(chi2, ir0), C));
  const FF g = ff_sub(dtf, ff_mul(ff_mul(chi2, chi), ff_mul(S, K.isq)));
  FF nx[3];
  for (int a = 0; a < 3; ++a) nx[a] = ff_add(ff_mul(f, x[a]), ff_mul(g, v[a]));
  const FF ir = ff_rsqrt(
      ff_add(ff_add(ff_mul(nx[0], nx[0]), ff_mul(nx[1], nx[1])), ff_mul(nx[2], nx[2])));
  const FF fd = ff_mul(ff_mul(ff_mul(K.sq, ir), ir0),
                       ff_mul(ff_sub(ff_mul(z, S), ff_c(1.0f, 0.0f)), chi));
  const FF gd = ff_sub(ff_c(1.0f, 0.0f), ff_mul(ff_mul(chi2, ir), C));
  for (int a = 0; a < 3; ++a) {
    const FF nv = ff_add(ff_mul(fd, x[a]), ff_mul(gd, v[a]));
    X[a] = ff_to_double(nx[a]);
    V[a] = ff_to_double(nv);
  }
  return true;
}

__device__ __forceinline__ KepFF kep_ff(const KepConst &K) {
  return {ff_split(K.sq), ff_split(K.isq), ff_split(K.imu)};
}

template <bool MIXED>
__global__ void k_kepler(const int64_t *d_nsingle, const int32_t *singles,
                         p3t_particles p, double dt, KepConst K, DevStatus *st) {
  pdl_wait();
  const int64_t ns = *d_nsingle;
  KepFF KF;
  if constexpr (MIXED) KF = kep_ff(K);
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < ns;
       k += (int64_t)gridDim.x * blockDim.x) {
    const int32_t i = singles[k];
    double X[3] = {p.x[i], p.y[i], p.z[i]}, V[3] = {p.vx[i], p.vy[i], p.vz[i]};
    bool done = false;
    if constexpr (MIXED) done = kepler_ff(X, V, dt, KF);
    if (!done && !kepler_uv(X, V, dt, K)) dev_fail(st, P3T_ERR_TIMEOUT, 60, 0);
    p.x[i] = X[0]; p.y[i] = X[1]; p.z[i] = X[2];
    p.vx[i] = V[0]; p.vy[i] = V[1]; p.vz[i] = V[2];
  }
}

// every particle of p (p3t_kepler_drift)
template <bool MIXED>
__global__ void k_kepler_all(p3t_particles p, double dt, KepConst K, DevStatus *st) {
  pdl_wait();
  KepFF KF;
  if constexpr (MIXED) KF = kep_ff(K);
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < p.n;
       i += (int64_t)gridDim.x * blockDim.x) {
    double X[3] = {p.x[i], p.y[i], p.z[i]}, V[3] = {p.vx[i], p.vy[i], p.vz[i]};
    bool done = false;
    if constexpr (MIXED) done = kepler_ff(X, V, dt, KF);
    if (!done && !kepler_uv(X, V, dt, K)) dev_fail(st, P3T_ERR_TIMEOUT, 60, 0);
    p.x[i] = X[0]; p.y[i] = X[1]; p.z[i] = X[2];
    p.vx[i] = V[0]; p.vy[i] = V[1]; p.vz[i] = V[2];
  }
}

// ---- Hermite-4 with block steps (+ collisions), one block per cluster ------
// Clusters of up to hermite_warp_max members (8 by default) run one warp each,
// so that the FP64 instructions of their few work items are not spread over
// idle lanes of several warps (two to five members: integrate_five below);
// larger ones up to 128 members run one 128-thread block each, their work items (member components, or (active member, source)
// terms) dealt round-robin over the four warps so that one long cluster keeps
// the FP64 pipes of all four SM sub-partitions busy.  Each active member's
// force is the sum, in the fixed order star term first then sources in
// ascending index, of terms computed in parallel (state in shared memory) or,
// above 128 members, by one thread per member (state in a global workspace).
//
// Perfect accretion (Sec. 2.4.1; on when f_radius > 0 and physical
// radii are given): at every force evaluation each evaluated member records
// the lowest-index member outside its composite that it touches, r < f (R_k
// + R_j).  After the correction the touching members (with the composites
// they belong to) become one composite: centre-of-mass position and velocity
// at the block time, hard force and jerk the mass-weighted mean over the
// composite with its inner pairs left out, a first step eta0 |a| / |j|.  The
// dissipated energy is the change of the affected members' kinetic, star and
// pair energy (changeover functions replaced by unity, the cluster standing
// for the neighbours).  One thread does this bookkeeping in a fixed order;
// collisions are rare.
constexpr int kHMax = 128;  // largest cluster kept in shared memory
// the largest cluster integrated by one warp is a launch-shape choice
// (p3t_set_tuning; 8 by default): larger ones take a block of four warps,
// whose pair terms then run on four sub-partitions' FP64 pipes.  The one-warp
// kernel is compiled for clusters of up to 8, 16 and 32 members (its shared
// memory grows with the bound, so the smallest that fits is launched).
constexpr int32_t kNone = 0x7fffffff;  // no collision partner

template <int KM>
struct HSmall {  // a cluster of <= KM members
  double x[3][KM], v[3][KM], a[3][KM], j[3][KM];
  double p[3][KM], pv[3][KM];
  double a1[3][KM], j1[3][KM], a2e[3][KM], a3[3][KM];
  double m[KM], iro[KM], rp[KM];
  // one batch of pair terms: B = NT / (nc + 1) members x (nc + 1) terms, at
  // most NT (a batch is one pass of the block's threads), and at least the
  // nc + 1 terms of one member
  static constexpr int kT = KM + 1 > 32 ? KM + 1 : 32;
  double T[kT][6];
  int64_t t[KM];
  int32_t lvl[KM], act[KM], set[KM], nset[KM], partner[KM], chg[KM];
};

static_assert(sizeof(HSmall<kHMax>) <= 48 * 1024,
              "HSmall must fit the default dynamic shared memory");

struct HCtl {  // per-block control, shared memory
  int64_t red[2][4];
  int32_t wcount[4];
  int64_t cluster;
  int nact, any, ncomp, stop;
  double edisp;
};

template <int KM>
struct SmallView {
  HSmall<KM> *S;
  static constexpr bool kBig = false;
  __device__ double &x(int q, int k) const { return S->x[q][k]; }
  __device__ double &v(int q, int k) const { return S->v[q][k]; }
  __device__ double &a(int q, int k) const { return S->a[q][k]; }
  __device__ double &j(int q, int k) const { return S->j[q][k]; }
  __device__ double &p(int q, int k) const { return S->p[q][k]; }
  __device__ double &pv(int q, int k) const { return S->pv[q][k]; }
  __device__ double &a1(int q, int k) const { return S->a1[q][k]; }
  __device__ double &j1(int q, int k) const { return S->j1[q][k]; }
  __device__ double &a2e(int q, int k) const { return S->a2e[q][k]; }
  __device__ double &a3(int q, int k) const { return S->a3[q][k]; }
  __device__ double &m(int k) const { return S->m[k]; }
  __device__ double &iro(int k) const { return S->iro[k]; }
  __device__ double &rp(int k) const { return S->rp[k]; }
  __device__ int64_t &t(int k) const { return S->t[k]; }
  __device__ int32_t &lvl(int k) const { return S->lvl[k]; }
  __device__ int32_t &act(int k) const { return S->act[k]; }
  __device__ int32_t &set(int k) const { return S->set[k]; }
  __device__ int32_t &nset(int k) const { return S->nset[k]; }
  __device__ int32_t &partner(int k) const { return S->partner[k]; }
  __device__ int32_t &chg(int k) const { return S->chg[k]; }
};

// global workspace of the large clusters: 33 double, 1 int64 and 6 int32
// arrays of cap entries, a cluster's members at its member offset
struct HBig {
  double *d;
  int64_t *t;
  int32_t *i;
  int64_t cap;
};
struct BigView {
  double *d;
  int64_t *tt;
  int32_t *ii;
  int64_t cap, off;
  static constexpr bool kBig = true;
  __device__ double &D(int arr, int k) const { return d[arr * cap + off + k]; }
  __device__ int32_t &I(int arr, int k) const { return ii[arr * cap + off + k]; }
  __device__ double &x(int q, int k) const { return D(q, k); }
  __device__ double &v(int q, int k) const { return D(3 + q, k); }
  __device__ double &a(int q, int k) const { return D(6 + q, k); }
  __device__ double &j(int q, int k) const { return D(9 + q, k); }
  __device__ double &p(int q, int k) const { return D(12 + q, k); }
  __device__ double &pv(int q, int k) const { return D(15 + q, k); }
  __device__ double &a1(int q, int k) const { return D(18 + q, k); }
  __device__ double &j1(int q, int k) const { return D(21 + q, k); }
  __device__ double &a2e(int q, int k) const { return D(24 + q, k); }
  __device__ double &a3(int q, int k) const { return D(27 + q, k); }
  __device__ double &m(int k) const { return D(30, k); }
  __device__ double &iro(int k) const { return D(31, k); }
  __device__ double &rp(int k) const { return D(32, k); }
  __device__ int64_t &t(int k) const { return tt[off + k]; }
  __device__ int32_t &lvl(int k) const { return I(0, k); }
  __device__ int32_t &act(int k) const { return I(1, k); }
  __device__ int32_t &set(int k) const { return I(2, k); }
  __device__ int32_t &nset(int k) const { return I(3, k); }
  __device__ int32_t &partner(int k) const { return I(4, k); }
  __device__ int32_t &chg(int k) const { return I(5, k); }
};

// composites handed to the kick and the merge (Sec. 2.4.1)
struct CollOut {
  unsigned long long *ctr;  // (records << 32) | entries
  int4 *ent;                // {particle, lowest member of its composite, lo, hi}
  int4 *rec;                // {cluster label, first entry, entries, 0}
  double *rec_e;            // energy dissipated in the cluster
  int32_t *slot;            // particle -> its entry, or -1
  int64_t ent_cap, rec_cap;
};

// x 2^k and ilogb(x) read from and written to the exponent field with integer
// operations when x (and the result) are normal -- the same values as ldexp
// and ilogb, without an FP64 instruction (one costs 64 cycles of a
// sub-partition's FP64 pipe on this part) -- and by ldexp / ilogb otherwise.
// The step estimates only choose a power-of-two step: formed in FP32 from
// components scaled by an exact power of two 2^k (j by s, a2 by s^2, a3 by
// s^3, s = 2^e close to the step) so that nothing overflows FP32.
__device__ __forceinline__ float norm3f(double a, double b, double c, int k) {
  const float x = d2f_scaled(a, k), y = d2f_scaled(b, k), z = d2f_scaled(c, k);
  return sqrtf(x * x + y * y + z * z);
}

// largest dt / 2^lvl not above dt_des, at most twice the previous step, and
// commensurate with the current time t (units of dt / 2^40).  The search
// starts at a lower bound from the binary exponents and t's trailing zeros
// give the commensurability level directly; the result is the same as
// stepping lvl up one at a time.
__device__ __forceinline__ int quantise_level(double dt_des, double dt, int prev,
                                              int64_t t, bool &underflow) {
  int lvl = 0;
  const long long bd = __double_as_longlong(dt), bs = __double_as_longlong(dt_des);
  const int edt = (int)((bd >> 52) & 0x7ff);
  if (bd > 0 && edt > P3T_KMAX && edt < 0x7ff &&
      (bs & 0x7fffffffffffffffLL) <= 0x7ff0000000000000LL) {
    // dt positive and normal down to dt / 2^KMAX, dt_des not NaN: as integers
    // the bit patterns order like the values (negative dt_des, -0 included,
    // below every positive one), and dt / 2^l is dt's pattern less l << 52
    if (bs > 0 && bs < bd) {
      int l0 = ilogb_fast(dt) - ilogb_fast(dt_des) - 1;  // dt / 2^l > dt_des for l <= l0
      lvl = l0 < 0 ? 0 : (l0 > P3T_KMAX ? P3T_KMAX : l0);
    }
    while (lvl < P3T_KMAX && bd - ((long long)lvl << 52) > bs) ++lvl;
    if (bd - ((long long)lvl << 52) > bs) underflow = true;
  } else {
    if (dt_des > 0.0 && dt_des < dt) {
      int l0 = ilogb(dt) - ilogb(dt_des) - 1;
      lvl = l0 < 0 ? 0 : (l0 > P3T_KMAX ? P3T_KMAX : l0);
    }
    while (lvl < P3T_KMAX && ldexp(dt, -lvl) > dt_des) ++lvl;
    if (ldexp(dt, -lvl) > dt_des) underflow = true;
  }
  if (lvl < prev - 1) lvl = prev - 1;
  if (t != 0) {
    const int need = P3T_KMAX - __ffsll((long long)t) + 1;  // 2^(40-lvl) must divide t
    if (lvl < need) lvl = need;
  }
  return lvl > P3T_KMAX ? P3T_KMAX : lvl;
}

// first step eta0 |a| / |j| = (eta0 |a| / |j s|) s, s = 2^e
template <class V>
__device__ __forceinline__ int first_level(const V &S, int k, const p3t_params &prm, double dt,
                                           int64_t t, bool &underflow) {
  const int e = ilogb_fast(dt);
  const float an = norm3f(S.a(0, k), S.a(1, k), S.a(2, k), 0);
  const float jn = norm3f(S.j(0, k), S.j(1, k), S.j(2, k), e);
  const double dtd = jn > 0.0f ? ldexp_fast(f2d_exact((float)prm.eta0 * an / jn), e) : dt;
  return quantise_level(dtd, dt, 0, t, underflow);
}

// term of source j (j == nc: the star) on member k at the block-time state
// (p, pv): the (1 - K) pair force and its jerk (Eq. hardforce), one
// reciprocal square root per pair, 1/max(r_out) taken as min(1/r_out).  The
// star is a source at the origin, at rest, of mass M_*, with 1/r_out = 0 (so
// y = 0: no changeover): the same instructions then give exactly the star
// term -G M_* x / |x|^3 and its jerk, with no divergent path.  Members of k's
// own composite are left out; with `detect`, hit reports contact r < f (R_k +
// R_j) with another member.
template <class V>
__device__ __forceinline__ void hard_term(const V &S, int nc, int k, int j,
                                          const p3t_params &prm, double i1mg, bool detect,
                                          double out[6], bool &hit) {
  for (int q = 0; q < 6; ++q) out[q] = 0.0;
  hit = false;
  const bool star = j == nc;
  if (!star && (j == k || S.set(j) == S.set(k))) return;
  const int js = star ? k : j;  // an index that can be read
  const double xk = S.p(0, k), yk = S.p(1, k), zk = S.p(2, k);
  const double vxk = S.pv(0, k), vyk = S.pv(1, k), vzk = S.pv(2, k);
  const double rx = xk - (star ? 0.0 : S.p(0, js)), ry = yk - (star ? 0.0 : S.p(1, js)),
               rz = zk - (star ? 0.0 : S.p(2, js));
  const double ux = vxk - (star ? 0.0 : S.pv(0, js)), uy = vyk - (star ? 0.0 : S.pv(1, js)),
               uz = vzk - (star ? 0.0 : S.pv(2, js));
  const double r2 = __fma_rn(rx, rx, __fma_rn(ry, ry, rz * rz));
  if (detect && !star) {
    const double sr = prm.f_radius * (S.rp(k) + S.rp(js));
    hit = r2 < sr * sr;
  }
  if (r2 == 0.0) return;
  const double rinv = rsqrt(r2);
  const double r = r2 * rinv;
  const double irot = star ? 0.0 : (S.iro(k) < S.iro(js) ? S.iro(k) : S.iro(js));
  const double yv = r * irot;
  if (yv >= 1.0) return;
  double w = 1.0, dK = 0.0;
  if (yv > prm.gamma) {
    const double xs = (yv - prm.gamma) * i1mg;
    const double x2 = xs * xs, x3 = x2 * xs, x4 = x2 * x2, u = 1.0 - xs;
    w = 1.0 - x4 * (35.0 - 84.0 * xs + 70.0 * x2 - 20.0 * x3);
    dK = 140.0 * x3 * (u * u * u) * i1mg;
  }
  const double rinv2 = rinv * rinv;
  const double g3 = prm.G * (star ? prm.m_star : S.m(js)) * (rinv2 * rinv);
  const double f = g3 * w;
  const double rv = __fma_rn(rx, ux, __fma_rn(ry, uy, rz * uz));
  out[0] = f * rx; out[1] = f * ry; out[2] = f * rz;
  const double c = __fma_rn(dK * rv * rinv, irot, 3.0 * w * rv * rinv2);
  out[3] = g3 * __fma_rn(-c, rx, w * ux);
  out[4] = g3 * __fma_rn(-c, ry, w * uy);
  out[5] = g3 * __fma_rn(-c, rz, w * uz);
}

// the members with pred(k), ascending, into act[0..); returns their number
template <int NT, class V, class Pred>
__device__ int build_list(const V &S, HCtl &C, int nc, Pred pred) {
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  int base = 0;
  for (int c0 = 0; c0 < nc; c0 += NT) {
    const int k = c0 + tid;
    const bool on = k < nc && pred(k);
    const unsigned bal = __ballot_sync(0xffffffffu, on);
    if (lane == 0) C.wcount[warp] = __popc(bal);
    __syncthreads();
    int off = base, tot = 0;
    for (int q = 0; q < NT / 32; ++q) {
      if (q < warp) off += C.wcount[q];
      tot += C.wcount[q];
    }
    if (on) S.act(off + __popc(bal & ((1u << lane) - 1u))) = k;
    base += tot;
    __syncthreads();
  }
  return base;
}

// forces on the listed members act[0..nact) from (p, pv) into (a1, j1); with
// `detect`, each one's lowest touching partner into partner[]; then the
// composites' mean force
template <int NT, class V>
__device__ void block_forces(const V &S, HCtl &C, double (*Tb)[6], int nc, int nact, int item,
                             const p3t_params &prm, double i1mg, bool detect) {
  if constexpr (!V::kBig) {
    const int per = nc + 1;
    const int B = NT / per > 0 ? NT / per : 1;  // members per batch
    for (int b0 = 0; b0 < nact; b0 += B) {
      const int nb = min(B, nact - b0);
      const int items = nb * per;
      for (int i = item; i < items; i += NT) {
        const int bm = i / per, jj = i - bm * per;
        const int k = S.act(b0 + bm);
        bool hit;
        hard_term(S, nc, k, jj, prm, i1mg, detect, Tb[i], hit);
        if (hit) atomicMin(&S.partner(k), jj);
      }
      __syncthreads();
      for (int i = item; i < nb * 6; i += NT) {
        const int bm = i / 6, q = i - bm * 6;
        const int k = S.act(b0 + bm);
        const int base = bm * per;
        double acc = 0.0;
        acc -= Tb[base + nc][q];
        for (int jj = 0; jj < nc; ++jj) acc -= Tb[base + jj][q];
        if (q < 3) S.a1(q, k) = acc; else S.j1(q - 3, k) = acc;
      }
      __syncthreads();
    }
  } else {
    for (int b = threadIdx.x; b < nact; b += NT) {
      const int k = S.act(b);
      double acc[6], out[6];
      bool hit;
      hard_term(S, nc, k, nc, prm, i1mg, false, out, hit);
      for (int q = 0; q < 6; ++q) acc[q] = 0.0 - out[q];
      for (int jj = 0; jj < nc; ++jj) {
        hard_term(S, nc, k, jj, prm, i1mg, detect, out, hit);
        for (int q = 0; q < 6; ++q) acc[q] -= out[q];
        if (hit && S.partner(k) == kNone) S.partner(k) = jj;
      }
      for (int q = 0; q < 3; ++q) { S.a1(q, k) = acc[q]; S.j1(q, k) = acc[3 + q]; }
    }
    __syncthreads();
  }
  if (C.ncomp) {
    // composite force: sum_l m_l a_l / sum_l m_l, ascending l (sets of >= 2)
    for (int b = item; b < nact; b += NT) {
      const int r = S.act(b);
      if (S.set(r) != r) continue;
      int size = 0;
      double M = 0.0, A[3] = {0, 0, 0}, J[3] = {0, 0, 0};
      for (int l = 0; l < nc; ++l) {
        if (S.set(l) != r) continue;
        ++size;
        M += S.m(l);
        for (int q = 0; q < 3; ++q) { A[q] += S.m(l) * S.a1(q, l); J[q] += S.m(l) * S.j1(q, l); }
      }
      if (size < 2) continue;
      for (int l = 0; l < nc; ++l) {
        if (S.set(l) != r) continue;
        for (int q = 0; q < 3; ++q) { S.a1(q, l) = A[q] / M; S.j1(q, l) = J[q] / M; }
      }
    }
    __syncthreads();
  }
}

// the block minima of two non-negative values (one warp: no shared memory)
template <int NT>
__device__ __forceinline__ void block_min2(int64_t &a, int64_t &b, int64_t (*red)[4]) {
  a = warp_min64(a);
  b = warp_min64(b);
  if constexpr (NT > 32) {
    if ((threadIdx.x & 31) == 0) {
      red[0][threadIdx.x >> 5] = a;
      red[1][threadIdx.x >> 5] = b;
    }
    __syncthreads();
    int64_t ra = red[0][0], rb = red[1][0];
    for (int q = 1; q < NT / 32; ++q) {
      ra = red[0][q] < ra ? red[0][q] : ra;
      rb = red[1][q] < rb ? red[1][q] : rb;
    }
    __syncthreads();
    a = ra;
    b = rb;
  }
}

// energy of the members with chg & 1 as far as replacing them can change it:
// kinetic and star energy, and the pair energy of every pair with one end
// among them (once), pairs in one set left out; state (p, pv)
template <class V>
__device__ double set_energy(const V &S, int nc, bool new_sets, const p3t_params &prm) {
  double E = 0.0;
  for (int k = 0; k < nc; ++k) {
    if (!(S.chg(k) & 1)) continue;
    const double vx = S.pv(0, k), vy = S.pv(1, k), vz = S.pv(2, k);
    const double x = S.p(0, k), y = S.p(1, k), z = S.p(2, k);
    E += 0.5 * S.m(k) * (vx * vx + vy * vy + vz * vz);
    E -= prm.G * prm.m_star * S.m(k) / sqrt(x * x + y * y + z * z);
  }
  for (int k = 0; k < nc; ++k) {
    if (!(S.chg(k) & 1)) continue;
    const int sk = new_sets ? S.set(k) : S.nset(k);
    for (int l = 0; l < nc; ++l) {
      const int sl = new_sets ? S.set(l) : S.nset(l);
      if (l == k || ((S.chg(l) & 1) && l < k) || sl == sk) continue;
      const double dx = S.p(0, k) - S.p(0, l), dy = S.p(1, k) - S.p(1, l),
                   dz = S.p(2, k) - S.p(2, l);
      const double r2 = dx * dx + dy * dy + dz * dz;
      if (r2 == 0.0) continue;
      E -= prm.G * S.m(k) * S.m(l) / sqrt(r2);
    }
  }
  return E;
}

// one thread: joins the touching members into composites at block time tn.
// On entry (p, pv) hold every member's state at tn; nset holds the sets
// before, set receives the sets after.
template <class V>
__device__ void collide_serial(const V &S, HCtl &C, int nc, int64_t tn, const p3t_params &prm) {
  for (int k = 0; k < nc; ++k) S.nset(k) = S.set(k);
  for (int k = 0; k < nc; ++k) {
    if (S.partner(k) == kNone) continue;
    const int ra = S.set(k), rb = S.set(S.partner(k));
    const int lo = ra < rb ? ra : rb, hi = ra < rb ? rb : ra;
    for (int l = 0; l < nc; ++l)
      if (S.set(l) == hi) S.set(l) = lo;
  }
  for (int k = 0; k < nc; ++k) S.chg(k) = 0;
  for (int k = 0; k < nc; ++k)
    if (S.partner(k) != kNone) S.chg(S.set(k)) = 2;
  for (int k = 0; k < nc; ++k)
    if (S.chg(S.set(k)) & 2) S.chg(k) |= 1;
  const double Eb = set_energy(S, nc, false, prm);  // sets before (nset)
  for (int r = 0; r < nc; ++r) {
    if (!(S.chg(r) & 1) || S.set(r) != r) continue;
    double Ms = 0.0, Q[6] = {0, 0, 0, 0, 0, 0};
    for (int l = 0; l < nc; ++l) {
      if (S.set(l) != r) continue;
      Ms += S.m(l);
      for (int q = 0; q < 3; ++q) { Q[q] += S.m(l) * S.p(q, l); Q[3 + q] += S.m(l) * S.pv(q, l); }
    }
    for (int l = 0; l < nc; ++l) {
      if (S.set(l) != r) continue;
      for (int q = 0; q < 3; ++q) { S.p(q, l) = Q[q] / Ms; S.pv(q, l) = Q[3 + q] / Ms; }
    }
  }
  const double Ea = set_energy(S, nc, true, prm);
  C.edisp += Eb - Ea;
  for (int k = 0; k < nc; ++k) {
    if (!(S.chg(k) & 1)) continue;
    for (int q = 0; q < 3; ++q) { S.x(q, k) = S.p(q, k); S.v(q, k) = S.pv(q, k); }
    S.t(k) = tn;
  }
  C.ncomp = 1;
}

// one thread: the cluster's composites (sets of >= 2) to the global list
template <class V>
__device__ void emit_composites(const V &S, const HCtl &C, int nc, int64_t off,
                                const int32_t *cl_mem, const CollOut &co, DevStatus *st) {
  int ne = 0;
  for (int r = 0; r < nc; ++r) {
    if (S.set(r) != r) continue;
    int size = 0;
    for (int l = 0; l < nc; ++l) size += S.set(l) == r;
    if (size >= 2) ne += size;
  }
  if (ne == 0) return;
  const unsigned long long old =
      atomicAdd(co.ctr, (1ull << 32) | (unsigned long long)ne);
  const int64_t rec = (int64_t)(old >> 32), e0 = (int64_t)(old & 0xffffffffull);
  if (rec >= co.rec_cap || e0 + ne > co.ent_cap) {
    dev_fail(st, P3T_ERR_CAPACITY, 63, e0 + ne);
    return;
  }
  co.rec[rec] = make_int4(cl_mem[off], (int)e0, ne, 0);
  co.rec_e[rec] = C.edisp;
  int e = (int)e0;
  for (int r = 0; r < nc; ++r) {
    if (S.set(r) != r) continue;
    int size = 0;
    for (int l = 0; l < nc; ++l) size += S.set(l) == r;
    if (size < 2) continue;
    const int lo = e, hi = e + size;
    for (int l = 0; l < nc; ++l) {
      if (S.set(l) != r) continue;
      const int32_t i = cl_mem[off + l];
      co.ent[e] = make_int4(i, cl_mem[off + r], lo, hi);
      co.slot[i] = e;
      ++e;
    }
  }
}

// block-step integration of one cluster (the whole block takes part); with
// `resume` S holds the state after the evaluation at tn that found a contact
template <int NT, class V>
__device__ void integrate_cluster(const V &S, HCtl &C, double (*Tb)[6], int64_t off, int nc,
                                  const int32_t *cl_mem, const p3t_particles &p,
                                  const p3t_params &prm, const HConst &hc, double dt, bool coll,
                                  const CollOut &co, unsigned long long &steps,
                                  bool &underflow, DevStatus *st, int64_t iter_limit,
                                  int32_t *rec, bool resume, int64_t tn, int64_t iter) {
  const int tid = threadIdx.x;
  const int item = (tid & 31) * (NT / 32) + (tid >> 5);  // consecutive items -> different warps
  bool uf = false;  // a step of this cluster fell below dt / 2^40
  const int64_t T = ((int64_t)1) << P3T_KMAX;
  const double i1mg = hc.i1mg, unit = hc.unit;
  int nact = 0;
  if (tid == 0) { C.any = resume ? 1 : 0; C.ncomp = 0; C.stop = 0; C.edisp = 0.0; }
  if (!resume) {
    for (int k = item; k < nc; k += NT) {
      const int32_t i = cl_mem[off + k];
      S.x(0, k) = p.x[i]; S.x(1, k) = p.y[i]; S.x(2, k) = p.z[i];
      S.v(0, k) = p.vx[i]; S.v(1, k) = p.vy[i]; S.v(2, k) = p.vz[i];
      for (int q = 0; q < 3; ++q) { S.p(q, k) = S.x(q, k); S.pv(q, k) = S.v(q, k); }
      S.m(k) = p.m[i];
      S.iro(k) = 1.0 / p.r_out[i];
      S.rp(k) = coll ? p.r_phys[i] : 0.0;
      S.set(k) = k;
      S.partner(k) = kNone;
      if (rec) rec[i] = 0;
    }
  }
  __syncthreads();
  if (!resume) {
    // initial forces of every member (the block-time state is the initial
    // state), first steps
    nact = build_list<NT>(S, C, nc, [](int) { return true; });
    block_forces<NT>(S, C, Tb, nc, nact, item, prm, i1mg, coll);
    for (int k = item; k < nc; k += NT) {
      for (int q = 0; q < 3; ++q) { S.a(q, k) = S.a1(q, k); S.j(q, k) = S.j1(q, k); }
      S.t(k) = 0;
      S.lvl(k) = first_level(S, k, prm, dt, 0, uf);
      if (S.partner(k) != kNone) C.any = 1;
    }
    if (uf) C.stop = 1;
    __syncthreads();
  }
  for (;;) {
    // a step below dt / 2^40 ends the cluster's integration (the error is
    // recorded when the block finishes): every thread reads the flag after
    // the barrier that follows its last write
    if (C.stop) break;
    if (C.any) {
      // collisions found by the last evaluation: every member's state at tn
      for (int k = item; k < nc; k += NT)
        if (S.t(k) == tn)
          for (int q = 0; q < 3; ++q) { S.p(q, k) = S.x(q, k); S.pv(q, k) = S.v(q, k); }
      __syncthreads();
      if (tid == 0) collide_serial(S, C, nc, tn, prm);
      __syncthreads();
      nact = build_list<NT>(S, C, nc, [&](int k) { return (S.chg(k) & 1) != 0; });
      block_forces<NT>(S, C, Tb, nc, nact, item, prm, i1mg, false);
      for (int b = item; b < nact; b += NT) {
        const int k = S.act(b);
        for (int q = 0; q < 3; ++q) { S.a(q, k) = S.a1(q, k); S.j(q, k) = S.j1(q, k); }
        S.lvl(k) = first_level(S, k, prm, dt, tn, uf);
      }
      for (int k = item; k < nc; k += NT) S.partner(k) = kNone;
      if (uf) C.stop = 1;
      __syncthreads();
      if (tid == 0) C.any = 0;
      __syncthreads();
      if (C.stop) break;
    }
    int64_t e_min = T, t_min = T;
    for (int k = tid; k < nc; k += NT) {
      const int64_t e = S.t(k) + (T >> S.lvl(k));
      e_min = e < e_min ? e : e_min;
      t_min = S.t(k) < t_min ? S.t(k) : t_min;
    }
    block_min2<NT>(e_min, t_min, C.red);
    tn = e_min;
    const int64_t tmin = t_min;
    if (tmin >= T) break;
    if (++iter > iter_limit) {
      if (tid == 0) dev_fail(st, P3T_ERR_TIMEOUT, 61, 0);
      break;
    }
    // predict every member (component items)
    for (int i = item; i < nc * 3; i += NT) {
      const int k = i / 3, q = i - 3 * k;
      const double D = i2d_exact(tn - S.t(k)) * unit;
      const double jq = S.j(q, k), aq = S.a(q, k), vq = S.v(q, k);
      // Horner form, fused: x + D (v + D (a/2 + D j/6)), v + D (a + D j/2)
      // (the halvings exact, as exponent shifts)
      S.p(q, k) = __fma_rn(__fma_rn(__fma_rn(jq * (1.0 / 6.0), D, ldexp_fast(aq, -1)), D, vq),
                           D, S.x(q, k));
      S.pv(q, k) = __fma_rn(__fma_rn(ldexp_fast(jq, -1), D, aq), D, vq);
    }
    __syncthreads();
    nact = build_list<NT>(S, C, nc, [&](int k) { return S.t(k) + (T >> S.lvl(k)) == tn; });
    block_forces<NT>(S, C, Tb, nc, nact, item, prm, i1mg, coll);
    // correct (component items of the active members)
    for (int i = item; i < nact * 3; i += NT) {
      const int b = i / 3, q = i - 3 * b;
      const int k = S.act(b);
      const int lv = S.lvl(k), sh = P3T_KMAX - lv;
      const double D = ldexp_fast(unit, sh);
      // 1 / D = 2^lvl (1 / dt) exactly (D = dt 2^-lvl): a product, not a division
      const double iD2 = ldexp_fast(hc.idt2, 2 * lv), iD3 = ldexp_fast(hc.idt3, 3 * lv);
      const double da = S.a(q, k) - S.a1(q, k);
      const double j0 = S.j(q, k), j1 = S.j1(q, k);
      const double A2 = __fma_rn(-D, __fma_rn(2.0, j1, 4.0 * j0), -6.0 * da) * iD2;
      const double A3 = __fma_rn(6.0 * D, j0 + j1, 12.0 * da) * iD3;
      S.a2e(q, k) = __fma_rn(D, A3, A2);
      S.a3(q, k) = A3;
      const double c3 = ldexp_fast(hc.c3u, 3 * sh), c4 = ldexp_fast(hc.c4u, 4 * sh),
                   c5 = ldexp_fast(hc.c5u, 5 * sh);
      S.x(q, k) = __fma_rn(A3, c5, __fma_rn(A2, c4, S.p(q, k)));
      S.v(q, k) = __fma_rn(A3, c4, __fma_rn(A2, c3, S.pv(q, k)));
      S.a(q, k) = S.a1(q, k);
      S.j(q, k) = j1;
    }
    __syncthreads();
    // new steps of the active members
    for (int b = item; b < nact; b += NT) {
      const int k = S.act(b);
      const double D = ldexp_fast(unit, P3T_KMAX - S.lvl(k));
      const int e = ilogb_fast(D);  // dt = sqrt(eta num_s / den_s) s
      const float an = norm3f(S.a(0, k), S.a(1, k), S.a(2, k), 0);
      const float jn = norm3f(S.j(0, k), S.j(1, k), S.j(2, k), e);
      const float a2n = norm3f(S.a2e(0, k), S.a2e(1, k), S.a2e(2, k), 2 * e);
      const float a3n = norm3f(S.a3(0, k), S.a3(1, k), S.a3(2, k), 3 * e);
      const float num = an * a2n + jn * jn, den = jn * a3n + a2n * a2n;
      const double dtd =
          den > 0.0f ? ldexp_fast(f2d_exact(sqrtf((float)prm.eta * num / den)), e) : dt;
      S.t(k) = tn;
      S.lvl(k) = quantise_level(dtd, dt, S.lvl(k), tn, uf);
      if (S.partner(k) != kNone) C.any = 1;
      if (rec) rec[cl_mem[off + k]] += 1;
    }
    if (uf) C.stop = 1;
    if (tid == 0) steps += (unsigned long long)nact;
    __syncthreads();
  }
  for (int k = item; k < nc; k += NT) {
    const int32_t i = cl_mem[off + k];
    p.x[i] = S.x(0, k); p.y[i] = S.x(1, k); p.z[i] = S.x(2, k);
    p.vx[i] = S.v(0, k); p.vy[i] = S.v(1, k); p.vz[i] = S.v(2, k);
  }
  if (tid == 0 && C.ncomp) emit_composites(S, C, nc, off, cl_mem, co, st);
  if (uf) underflow = true;
  __syncthreads();
}

// ---- one warp per cluster of two to five: FP64 slots shared by the lanes -------
// On this part an FP64 warp instruction holds its sub-partition's pipe for 64
// cycles whatever its mask (measured: 64.2 cycles a DFMA with 1 to 32 active
// lanes, in one chain or eight), so a block step of a small cluster costs its
// number of FP64 warp instructions and the latency of what stands between
// them, not its arithmetic.  Clusters of at most five members (nearly all)
// therefore keep a member in six lanes (three positions, three velocities;
// state, forces and times in registers), and independent operations sit in
// different lanes of one instruction: every FP64 slot is one fma(A, B, C) with
// operands chosen per lane, a product A B + 0, a difference fma(-1, B, C).
// Factors of two are moved between operands (exact), so every value has the
// bits of hard_term and integrate_cluster:
//  - predictor, 4 slots: D = RN(n unit) from one fma on 2^52 + n (beside j/3),
//    then positions and velocities side by side;
//  - pair terms, six lanes a term, five terms a round: r.r beside r.u; with
//    every term inside gamma r_out (decided on the leading bits, with a
//    margin: K = 0) the changeover is left out, otherwise its two polynomials
//    run side by side: 14 or 30 slots a round against 55 or 75 for hard_term's
//    one lane a term;
//  - corrector, 8 slots: A2 beside A3, then x beside v.
//  - step criterion: approximate FP32 norms decide the level unless they are
//    within 2^-14 of a power of two (then the criterion as written), so no
//    conversion, root or division of full precision is on the path.
// What bounds it: the FP64 pipe of one sub-partition, 27 to 44 slots of the
// 4,000-5,500 cycles of a block step.  Measured (one cluster, both members
// active): 6.5 -> 2.3 us a block step inside gamma r_out, 6.8 -> 3.0 us in the
// changeover; triples 5.8 -> 2.7 us; 20,000 pairs of 15 block steps at once
// 1,844 -> 641 us.  Clusters of 6 and more keep integrate_cluster's one lane a
// term (eight members: 25 rounds here against 3 batches there).
constexpr int kFive = 5;

struct HFive {
  double P[kFive + 1][6];   // positions and velocities at the block time; the star's row is zero
  double D[kFive][6];       // a round's r and u
  double T[kFive * kFive][6];
  double gm[kFive + 1], iro[kFive + 1];  // G m, 1 / r_out; the star: G M_*, 0
  double sr2[kFive * kFive];             // (f (R_k + R_j))^2
  float irf2[kFive + 1];                 // 1 / r_out^2 in FP32
  int32_t partner[kFive];
};

// (float)(x 2^k)
__device__ __forceinline__ float scaled_float(double x, int k) {
  const int hi = __double2hiint(x), e = (hi >> 20) & 0x7ff;
  const bool plain = (unsigned)(e - 1) < 2046u && (unsigned)(e + k - 1) < 2046u;
  return (float)(plain || k == 0 ? __hiloint2double(hi + (k << 20), __double2loint(x))
                                 : ldexp(x, k));
}

// the terms of the listed members (act: four bits each) at the block-time
// state F.P, five a round, into F.T[b nc + jj] (jj: the other members by
// index, then the star)
__device__ __forceinline__ void five_terms(HFive &F, int nc, int nact, unsigned act,
                                           const p3t_params &prm, const HConst &hc, bool coll) {
  const int lane = threadIdx.x & 31, g = lane / 6, c = lane - 6 * g, g0 = lane - c;
  const bool jerk = c >= 3, hlp = c == 1;
  const int terms = nact * nc;
  const unsigned inc = 65536u / (unsigned)nc + 1u;  // x / nc = x inc >> 16 for x <= 25
  for (int t0 = 0; t0 < terms; t0 += kFive) {
    const int ti = t0 + g;
    const bool in = g < kFive && ti < terms;
    const int tc = in ? ti : 0;
    const int b = (int)(((unsigned)tc * inc) >> 16), jj = tc - b * nc;
    const int k = (int)(act >> (4 * b)) & 7;
    const int j = jj == nc - 1 ? kFive : (jj < k ? jj : jj + 1);
    const double d = F.P[k][c] - F.P[j][c];
    const int gd = g < kFive ? g : 0;
    if (g < kFive) F.D[g][c] = d;
    const double Gm = F.gm[j], ik = F.iro[k], ij = F.iro[j];
    const double irot = __double_as_longlong(ik) < __double_as_longlong(ij) ? ik : ij;
    const float irf2 = fminf(F.irf2[k], F.irf2[j]);
    __syncwarp();
    const double rx = F.D[gd][0], ry = F.D[gd][1], rz = F.D[gd][2];
    const int o = jerk ? 3 : 0;
    // r.r in lanes 0-2, r.u in lanes 3-5
    const double s = __fma_rn(rx, F.D[gd][o], __fma_rn(ry, F.D[gd][o + 1], rz * F.D[gd][o + 2]));
    double r2 = shfl_d(s, g0);
    const int hi = __double2hiint(r2);
    if (coll && in && c == 0 && j < kFive && gt_pos(F.sr2[k * kFive + j], r2))
      atomicMin(&F.partner[k], j);
    const bool on = in && __double_as_longlong(r2) != 0;
    if (!on) r2 = 1.0;
    const double rinv = rsqrt(r2);
    // r^2 from its leading 20 bits (FP32 range checked by the exponent)
    const int e = hi >> 20;
    const float r2f = __uint_as_float(((unsigned)(e - 896) << 23) | ((unsigned)(hi & 0xfffff) << 3));
    const bool inner = !on || j == kFive || (e > 900 && e < 1100 && r2f * irf2 < hc.gin2);
    double w = 1.0, dK = 0.0;
    bool dead = false, any_mid = false;
    if (!__all_sync(0xffffffffu, inner)) {
      const double yv = (r2 * rinv) * irot;
      dead = ge_pos(yv, 1.0);
      const bool mid = on && !dead && gt_pos(yv, prm.gamma);
      any_mid = __any_sync(0xffffffffu, mid);
      if (any_mid) {
        // lanes 0, 2: w = 1 - x^4 P; lanes 3-5: dK; lane 1: P's first terms
        const double xs = (yv - prm.gamma) * hc.i1mg;
        const double v1 = __fma_rn(hlp ? 84.0 : xs, xs, 0.0);                          // x^2 | 84 x
        const double v2 = __fma_rn(hlp ? -1.0 : v1, hlp ? v1 : xs, hlp ? 35.0 : 0.0);  // x^3
        const double x2 = shfl_d(v1, g0);
        // x^4 | 1 - x | 70 x^2
        const double v3 = __fma_rn(hlp ? 70.0 : (jerk ? -1.0 : x2), jerk ? xs : x2,
                                   jerk ? 1.0 : 0.0);
        // 20 x^3 | u^2 | 35 - 84 x + 70 x^2
        const double v4 = __fma_rn(hlp ? 1.0 : (jerk ? v3 : 20.0), hlp ? v2 : (jerk ? v3 : v2),
                                   hlp ? v3 : 0.0);
        const double m4 = shfl_d(v4, g0 + 1);
        // P | u^3
        const double v5 = __fma_rn(jerk ? v4 : -1.0, jerk ? v3 : v4, jerk ? 0.0 : m4);
        // x^4 P | 140 x^3
        const double v6 = __fma_rn(jerk ? 140.0 : v3, jerk ? v2 : v5, 0.0);
        // w | 140 x^3 u^3
        const double v7 = __fma_rn(jerk ? v6 : -1.0, jerk ? v5 : v6, jerk ? 0.0 : 1.0);
        const double ww = shfl_d(v7, g0);
        const double dk = v7 * hc.i1mg;
        if (mid) {
          w = ww;
          dK = dk;  // read by the jerk lanes only
        }
      }
    }
    const double rq = F.D[gd][jerk ? c - 3 : c];
    const double m1 = (jerk ? 3.0 : rinv) * (jerk ? w : rinv);       // 3 w | rinv^2
    const double rinv2 = shfl_d(m1, g0);
    const double m2 = m1 * (jerk ? s : rinv);                        // 3 w r.u | rinv^3
    const double m3 = (jerk ? m2 : Gm) * (jerk ? rinv2 : m2);        // 3 w r.u rinv^2 | g3
    const double g3 = shfl_d(m3, g0);
    double out;
    if (!any_mid) {  // w = 1, dK = 0: f = g3, c = 3 r.u rinv^2
      out = g3 * (jerk ? __fma_rn(-m3, rq, d) : rq);
    } else {
      const double e1 = (jerk ? dK : g3) * (jerk ? s : w);           // dK r.u | f
      const double e2 = e1 * (jerk ? rinv : rq);                     // dK r.u rinv | f r
      const double t = __fma_rn(-__fma_rn(e2, irot, m3), rq, w * d);
      out = jerk ? g3 * t : e2;
    }
    if (in) F.T[ti][c] = on && !dead ? out : 0.0;
    __syncwarp();
  }
}

// the step criterion as first_level and integrate_cluster evaluate it: x1 = a
// and x2 = a2 in a member's position lanes, j and a3 in its velocity lanes
__device__ __forceinline__ double exact_step(double x1, double x2, bool vel, int other, int gq, int e,
                                          bool later, const HConst &hc, double dt) {
  const float n1 = sqrtf(norm_lanes(scaled_float(x1, vel ? e : 0), gq));
  const float n2 = sqrtf(norm_lanes(scaled_float(x2, vel ? 3 * e : 2 * e), gq));
  const float o1 = __shfl_sync(0xffffffffu, n1, other), o2 = __shfl_sync(0xffffffffu, n2, other);
  const float an = vel ? o1 : n1, jn = vel ? n1 : o1;
  const float a2n = vel ? o2 : n2, a3n = vel ? n2 : o2;
  const float num = an * a2n + jn * jn, den = later ? jn * a3n + a2n * a2n : jn;
  if (!(den > 0.0f)) return dt;
  return ldexp((double)(later ? sqrtf(hc.etaf * num / den) : hc.eta0f * an / jn), e);
}

// block-step integration of a cluster of 2..5 members by one warp: the values
// of integrate_cluster.  Returns true when done; when members touch (a
// composite is to be formed, rare) the state goes to S and *tn, and
// integrate_cluster carries on from there.
template <class V>
__device__ bool integrate_five(const V &S, HFive &F, int64_t off, int nc, const int32_t *cl_mem,
                               const p3t_particles &p, const p3t_params &prm, const HConst &hc,
                               double dt, bool coll, unsigned long long &steps, bool &underflow,
                               DevStatus *st, int64_t iter_limit, int32_t *rec, int64_t *tn_out,
                               int64_t *iter_out) {
  const int lane = threadIdx.x & 31, g = lane / 6, c = lane - 6 * g, q = c >= 3 ? c - 3 : c;
  const bool vel = c >= 3;
  const int other = g < kFive ? (vel ? lane - 3 : lane + 3) : lane;
  const int g0 = lane - c, gq = g0 + (vel ? 3 : 0);  // first lane of the member, of this half
  const bool mine = g < nc;
  const int64_t T = ((int64_t)1) << P3T_KMAX;
  const long long bd = __double_as_longlong(dt);
  const int e_unit = ((__double2hiint(hc.unit) >> 20) & 0x7ff) - 1023;
  // per-lane constants of the slots: positions | velocities
  const double b1 = vel ? 2.0 / 6.0 : hc.unit, o1 = vel ? -0.0 : hc.m52u;
  const double kap = vel ? 1.0 : 2.0, del = vel ? 12.0 : -6.0;
  const double gD0 = vel ? hc.unit6 : -2.0 * hc.unit, iD0 = vel ? hc.idt3 : hc.idt2;
  const double h0 = vel ? hc.c3u : hc.c4u, h1c = vel ? hc.c4u : hc.c5u;
  const int ni = vel ? 3 : 2, nh0 = vel ? 3 : 4, nh1 = vel ? 4 : 5;
  int32_t i = 0;
  double s0 = 0.0, vq = 0.0, a = 0.0, j = 0.0;
  if (mine) {
    i = cl_mem[off + g];
    const double *X = q == 0 ? p.x : (q == 1 ? p.y : p.z);
    const double *W = q == 0 ? p.vx : (q == 1 ? p.vy : p.vz);
    vq = W[i];
    s0 = vel ? vq : X[i];
    F.P[g][c] = s0;
    if (c == 0) {
      F.gm[g] = prm.G * p.m[i];
      F.partner[g] = kNone;
      if (rec) rec[i] = 0;
    }
    if (c == 1) {
      const double iro = 1.0 / p.r_out[i];
      const float f = (float)iro;
      F.iro[g] = iro;
      F.irf2[g] = f * f;
    }
  }
  if (lane < 6) F.P[kFive][lane] = 0.0;
  if (lane == 6) { F.gm[kFive] = hc.gms; F.iro[kFive] = 0.0; F.irf2[kFive] = 0.0f; }
  if (coll && lane < kFive * kFive) {
    const int k = lane / kFive, l = lane - kFive * k;
    if (k < nc && l < nc) {
      const double sr = prm.f_radius * (p.r_phys[cl_mem[off + k]] + p.r_phys[cl_mem[off + l]]);
      F.sr2[lane] = sr * sr;
    }
  }
  __syncwarp();
  bool uf = false, hit = false, done = true;
  int64_t t = 0, tn = 0, iter = 0;
  int lvl = 0, nact = nc;
  unsigned act = 0x43210;  // the active members, four bits each
  double pred = s0;
  int64_t e_end = 0;       // end of the member's step; the initial evaluation is at 0
  for (;;) {
    const bool on = mine && e_end == tn;
    five_terms(F, nc, nact, act, prm, hc, coll);
    // the fixed order: star, then the sources by index
    double a1 = 0.0, j1 = 0.0;
    {
      const unsigned bal = __ballot_sync(0xffffffffu, on && c == 0);
      const int b = on ? __popc(bal & ((1u << g0) - 1u)) : 0;
      const double *t = F.T[b * nc] + c;
      double acc = -t[6 * (nc - 1)] - t[0];
      if (nc > 2) acc -= t[6];
      if (nc > 3) acc -= t[12];
      if (nc > 4) acc -= t[18];
      const double oa = shfl_d(acc, other);
      a1 = vel ? oa : acc;
      j1 = vel ? acc : oa;
    }
    double A2 = 0.0, A3 = 0.0, a2e = 0.0;
    int e;  // the step criterion's scale 2^e
    if (iter > 0) {
      const int sh = P3T_KMAX - lvl;
      // A2 = (-D (2 j1 + 4 j0) - 6 da) / D^2, A3 = (6 D (j0 + j1) + 12 da) /
      // D^3 (the factor 2 of A2's sum moved to D, exactly)
      const double da = a - a1;
      const double sj = __fma_rn(kap, j, j1);
      const double A = __fma_rn(shift_exp(gD0, sh), sj, del * da) * shift_exp(iD0, ni * lvl);
      const double oA = shfl_d(A, other);
      A2 = vel ? oA : A;
      A3 = vel ? A : oA;
      const double h = __fma_rn(A2, shift_exp(h0, nh0 * sh), pred);
      const double sn = __fma_rn(A3, shift_exp(h1c, nh1 * sh), h);
      a2e = __fma_rn(shift_exp(hc.unit, sh), A3, A2);
      const double on_v = shfl_d(sn, other);
      if (on) {
        s0 = sn;
        vq = vel ? sn : on_v;
      }
      e = e_unit + sh;
    } else {
      e = e_unit + P3T_KMAX;
    }
    // the new step, first from squared norms of the components' leading 20 bits:
    // |a| and |a2| in the position lanes, |j| and |a3| in the velocity lanes;
    // where those do not decide its level, by the criterion as written
    double dtd;
    {
      const float x1 = lead_float(vel ? j1 : a1, vel ? e : 0);
      const float x2 = lead_float(vel ? A3 : a2e, vel ? 3 * e : 2 * e);
      const float n1 = norm_lanes(x1, gq), n2 = norm_lanes(x2, gq);
      const float o1 = __shfl_sync(0xffffffffu, n1, other),
                  o2 = __shfl_sync(0xffffffffu, n2, other);
      const float an = vel ? o1 : n1, jn = vel ? n1 : o1;  // squared
      const float a2n = vel ? o2 : n2, a3n = vel ? n2 : o2;
      const bool decided = step_estimate(an, jn, a2n, a3n, e, iter > 0, hc, bd, dtd);
      if (__any_sync(0xffffffffu, on && !decided))
        dtd = exact_step(vel ? j1 : a1, vel ? A3 : a2e, vel, other, gq, e, iter > 0, hc, dt);
    }
    if (on) {
      lvl = level_bits(dtd, bd, iter > 0 ? lvl : 0, tn, uf);
      a = a1;
      j = j1;
      t = tn;
      if (iter > 0 && rec && c == 0) rec[i] += 1;
      if (coll) hit = F.partner[g] != kNone;
    }
    if (iter > 0) steps += lane == 0 ? (unsigned long long)nact : 0ull;
    if (__any_sync(0xffffffffu, uf || hit)) {
      if (__any_sync(0xffffffffu, uf)) break;  // a step below dt / 2^40 ends the integration
      done = false;
      break;
    }
    // every step ends at or before T, so all members are at T once a block
    // time was T
    if (tn >= T) break;
    e_end = mine ? t + (T >> lvl) : T;
    tn = warp_min64(e_end < T ? e_end : T);
    if (++iter > iter_limit) {
      if (lane == 0) dev_fail(st, P3T_ERR_TIMEOUT, 61, 0);
      break;
    }
    // predict: x + D (v + D (a/2 + D j/6)), v + D (a + D j/2), with D = RN(n
    // unit) = fma(2^52 + n, unit, -2^52 unit) for the n units since t, and
    // the halves moved to D (exact)
    const long long n = tn - t;
    const double mg = __longlong_as_double(0x4330000000000000LL + n);
    const double s1 = __fma_rn(vel ? j : mg, b1, o1);
    const double os = shfl_d(s1, other);
    const double D = vel ? os : s1, Dh = shift_exp(D, -1);
    const double s2 = __fma_rn(vel ? j : os, vel ? Dh : D, a);
    const double s3 = __fma_rn(s2, vel ? D : Dh, vq);
    const double s4 = __fma_rn(s3, D, s0);
    pred = vel ? s3 : s4;
    if (mine) F.P[g][c] = pred;
    const unsigned bal = __ballot_sync(0xffffffffu, mine && e_end == tn && c == 0);
    act = 0;
    nact = 0;
#pragma unroll
    for (int m = 0; m < kFive; ++m)
      if ((bal >> (6 * m)) & 1u) { act |= (unsigned)m << (4 * nact); ++nact; }
    __syncwarp();
  }
  if (done) {
    if (mine) {
      double *X = q == 0 ? p.x : (q == 1 ? p.y : p.z);
      double *W = q == 0 ? p.vx : (q == 1 ? p.vy : p.vz);
      (vel ? W : X)[i] = s0;
    }
  } else if (mine) {
    (vel ? S.v(q, g) : S.x(q, g)) = s0;
    (vel ? S.pv(q, g) : S.p(q, g)) = pred;
    (vel ? S.j(q, g) : S.a(q, g)) = vel ? j : a;
    if (c == 0) {
      S.m(g) = p.m[i];
      S.iro(g) = F.iro[g];
      S.rp(g) = p.r_phys[i];
      S.set(g) = g;
      S.partner(g) = F.partner[g];
      S.t(g) = t;
      S.lvl(g) = lvl;
    }
  }
  *tn_out = tn;
  *iter_out = iter;
  if (uf) underflow = true;
  __syncwarp();
  return done;
}

// clusters of nc_lo..nc_hi members; NT threads per block; state in shared
// memory for up to KM members or (BIG) in the global workspace.  One block
// per cluster, clusters handed out dynamically (a long encounter keeps its
// block while the others move on).
template <int NT, int KM, bool BIG>
__global__ void __launch_bounds__(NT, NT == 32 ? 20 : 1) k_hermite_block(
    const int64_t *d_ncl, const int64_t *cl_off, const int32_t *cl_mem, p3t_particles p,
    p3t_params prm, HConst hc, double dt, int nc_lo, int nc_hi, unsigned long long *steps_out,
    int64_t *cursor, const int32_t *list, const int64_t *d_nlist, HBig big, CollOut co,
    DevStatus *st, int64_t iter_limit, int32_t *rec) {
  pdl_wait();
  __shared__ HCtl C;
  extern __shared__ __align__(16) unsigned char hsm[];
  static_assert(BIG || HSmall<KM>::kT >= NT, "a batch of pair terms must fit HSmall::T");
  HSmall<KM> *Sm = reinterpret_cast<HSmall<KM> *>(hsm);
  const int tid = threadIdx.x;
  // every cluster, or (list) the clusters of this kernel's sizes
  const int64_t ncl = list ? *d_nlist : *d_ncl;
  const bool coll = prm.f_radius > 0.0 && p.r_phys != nullptr;
  unsigned long long steps = 0;
  bool underflow = false;
  for (int64_t k = blockIdx.x;; k += gridDim.x) {
    // clusters of up to 128 members are handed out by a cursor (a long
    // encounter keeps its block while the others move on); the rare larger
    // ones are dealt statically
    int64_t c = k;
    if constexpr (NT == 32) {
      unsigned long long u = 0;
      if (tid == 0) u = atomicAdd(reinterpret_cast<unsigned long long *>(cursor), 1ull);
      c = (int64_t)__shfl_sync(0xffffffffu, u, 0);
    } else if constexpr (!BIG) {
      if (tid == 0) C.cluster = atomicAdd(reinterpret_cast<unsigned long long *>(cursor), 1ull);
      __syncthreads();
      c = C.cluster;
      __syncthreads();
    }
    if (c >= ncl) break;
    if (list) c = list[c];
    const int64_t off = cl_off[c];
    const int nc = (int)(cl_off[c + 1] - off);
    if (nc < nc_lo || nc > nc_hi) continue;
    if constexpr (BIG) {
      const BigView S{big.d, big.t, big.i, big.cap, off};
      integrate_cluster<NT>(S, C, nullptr, off, nc, cl_mem, p, prm, hc, dt, coll, co, steps,
                            underflow, st, iter_limit, rec, false, 0, 0);
    } else {
      const SmallView<KM> S{Sm};
      bool resume = false;
      int64_t tn = 0, iter = 0;
      if constexpr (NT == 32) {
        __shared__ HFive F;
        if (nc <= kFive && hc.fast) {
          if (integrate_five(S, F, off, nc, cl_mem, p, prm, hc, dt, coll, steps, underflow, st,
                             iter_limit, rec, &tn, &iter))
            continue;
          resume = true;
        }
      }
      integrate_cluster<NT>(S, C, Sm->T, off, nc, cl_mem, p, prm, hc, dt, coll, co, steps,
                            underflow, st, iter_limit, rec, resume, tn, iter);
    }
  }
  if (underflow) dev_fail(st, P3T_ERR_DT_UNDERFLOW, 62, 0);
  if (tid == 0 && steps_out && steps) atomicAdd(steps_out, steps);
}

// the step count and the Hermite kernels' cursors and list lengths to zero
__global__ void k_zero_hard(unsigned long long *steps, int64_t *p) {
  pdl_wait();
  if (threadIdx.x < 5) p[threadIdx.x] = 0;
  if (threadIdx.x == 5) *steps = 0ull;
}

// the clusters of more than hw members: up to kHMax into list[0..), larger
// ones into list[cap..); their numbers into n[0], n[1] (zeroed before).  The
// order within a list is arrival order: each cluster is integrated on its own,
// so the results do not depend on it.
__global__ void k_cluster_classes(const int64_t *d_ncl, const int64_t *cl_off, int hw,
                                  int64_t cap, int32_t *list, int64_t *n) {
  pdl_wait();
  const int64_t ncl = *d_ncl;
  for (int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; c < ncl;
       c += (int64_t)gridDim.x * blockDim.x) {
    const int64_t nc = cl_off[c + 1] - cl_off[c];
    if (nc <= hw) continue;
    const int big = nc > kHMax ? 1 : 0;
    const int64_t slot = (int64_t)atomicAdd(reinterpret_cast<unsigned long long *>(&n[big]), 1ull);
    if (slot < cap) list[big * cap + slot] = (int32_t)c;
  }
}

// ---- energy ----------------------------------------------------------------
__device__ __forceinline__ void two_sum_f(float &hi, float &lo, float b) {
  const float s = hi + b;
  const float bb = s - hi;
  lo += (hi - (s - bb)) + (b - bb);
  hi = s;
}

struct D4 {
  double x, y, z, w;
};
constexpr int kETile = 256;                // targets and sources of a tile
constexpr int kEThreads = kETile / 2;      // two targets a thread
constexpr int64_t kEBlocks = 152 * 4 * 8;  // blocks asked for: eight waves of four an SM

// E = sum m v^2/2 - sum G M m / r - sum_{i < j} G m_i m_j / r_ij.  Bound by the
// FP32 (FP64) pipe, so every pair of tiles is taken once (the pairs inside a
// tile twice at half weight): tile row I has the source tiles J >= I, and rows
// I and T - 1 - I together always T + 1, cut into chunks of equal length over
// blockIdx.y.  Mixed: a thread's two targets are the halves of packed FP32
// pairs (17 packed instructions for two pairs); FP64: 12 instructions a pair
// with 1 / r from the 20-bit seed.  Sources are staged by tile, a tile's sum
// in FP32 (FP64) per target, the tiles' sums in float-float (FP64).  Measured
// (one scalar target a thread over all sources before): mixed N = 1e5 11,640 ->
// 2,790 us, 1e4 703 -> 69; FP64 N = 1e4 10,950 -> 1,330.  (With rsqrtf
// for rsqrt_normal: 3,490 and 72.)
template <bool MIXED>
__global__ void __launch_bounds__(kEThreads) k_energy(p3t_particles p, p3t_params prm, int tiles,
                                                      int chunk, double *part) {
  pdl_wait();
  using V = typename std::conditional<MIXED, float4, D4>::type;
  __shared__ V s_h[kETile];
  __shared__ float4 s_l[MIXED ? kETile : 1];
  __shared__ double s_red[3][kEThreads / 32];
  const int64_t n = p.n;
  const int tid = threadIdx.x;
  double ek = 0.0, es = 0.0, ep = 0.0;
  const int rowA = blockIdx.x, rowB = tiles - 1 - rowA;
  const int lenA = tiles - rowA, len = rowA == rowB ? lenA : tiles + 1;
  const int p0 = blockIdx.y * chunk, p1 = min(len, p0 + chunk);
  for (int seg = 0; seg < 2; ++seg) {
    const int row = seg ? rowB : rowA;
    const int j0 = seg ? row + max(p0 - lenA, 0) : row + p0;
    const int j1 = seg ? row + (p1 - lenA) : row + min(p1, lenA);
    if (j0 >= j1) continue;
    double X[2], Y[2], Z[2], M[2];
    float xh[2], yh[2], zh[2], xl[2], yl[2], zl[2];
#pragma unroll
    for (int t = 0; t < 2; ++t) {
      const int64_t i = (int64_t)row * kETile + t * kEThreads + tid;
      X[t] = Y[t] = Z[t] = M[t] = 0.0;
      if (i < n) {
        X[t] = p.x[i]; Y[t] = p.y[i]; Z[t] = p.z[i]; M[t] = p.m[i];
        if (j0 == row) {
          ek += 0.5 * M[t] * (p.vx[i] * p.vx[i] + p.vy[i] * p.vy[i] + p.vz[i] * p.vz[i]);
          es += -prm.G * prm.m_star * M[t] / sqrt(X[t] * X[t] + Y[t] * Y[t] + Z[t] * Z[t]);
        }
      }
      if constexpr (MIXED) {
        split_f32(X[t], xh[t], xl[t]);
        split_f32(Y[t], yh[t], yl[t]);
        split_f32(Z[t], zh[t], zl[t]);
      }
    }
    f2 TX = 0, TY = 0, TZ = 0, TXL = 0, TYL = 0, TZL = 0;
    if constexpr (MIXED) {
      TX = f2_pk(xh[0], xh[1]); TY = f2_pk(yh[0], yh[1]); TZ = f2_pk(zh[0], zh[1]);
      TXL = f2_pk(xl[0], xl[1]); TYL = f2_pk(yl[0], yl[1]); TZL = f2_pk(zl[0], zl[1]);
    }
    float sh[2] = {0.f, 0.f}, sl[2] = {0.f, 0.f};
    double sd[2] = {0.0, 0.0};
    for (int J = j0; J < j1; ++J) {
      __syncthreads();
#pragma unroll
      for (int t = 0; t < 2; ++t) {
        const int q = t * kEThreads + tid;
        const int64_t j = (int64_t)J * kETile + q;
        const bool on = j < n;
        const double x = on ? p.x[j] : 0.0, y = on ? p.y[j] : 0.0, z = on ? p.z[j] : 0.0,
                     m = on ? p.m[j] : 0.0;
        if constexpr (MIXED) {
          float a, b, c, d, e, f, u, v;
          split_f32(x, a, d);
          split_f32(y, b, e);
          split_f32(z, c, f);
          split_f32(m, u, v);
          s_h[q] = make_float4(a, b, c, u);
          s_l[q] = make_float4(d, e, f, 0.f);
        } else {
          s_h[q].x = x; s_h[q].y = y; s_h[q].z = z; s_h[q].w = m;
        }
      }
      __syncthreads();
      const int lim = (int)min((int64_t)kETile, n - (int64_t)J * kETile);
      if constexpr (MIXED) {
        f2 b = 0ull;
#pragma unroll 4
        for (int q = 0; q < lim; ++q) {
          const float4 H = s_h[q], L = s_l[q];
          const f2 dx = add2(sub2(TX, f2_dup(H.x)), sub2(TXL, f2_dup(L.x)));
          const f2 dy = add2(sub2(TY, f2_dup(H.y)), sub2(TYL, f2_dup(L.y)));
          const f2 dz = add2(sub2(TZ, f2_dup(H.z)), sub2(TZL, f2_dup(L.z)));
          const f2 r2 = fma2(dx, dx, fma2(dy, dy, mul2(dz, dz)));
          const float ra = f2_lo(r2), rb = f2_hi(r2);
          f2 ri = f2_pk(rsqrt_normal(ra), rsqrt_normal(rb));
          if (!(ra >= 1.17549435e-38f && rb >= 1.17549435e-38f))  // zero or subnormal
            ri = f2_pk(ra > 0.f ? rsqrtf(ra) : 0.f, rb > 0.f ? rsqrtf(rb) : 0.f);
          // one Newton step
          const f2 c = fma2(mul2(f2_dup(-0.5f), r2), mul2(ri, ri), f2_dup(1.5f));
          b = fma2(f2_dup(H.w), mul2(ri, c), b);
        }
        const float w = J == row ? 0.5f : 1.0f;
        two_sum_f(sh[0], sl[0], f2_lo(b) * w);
        two_sum_f(sh[1], sl[1], f2_hi(b) * w);
      } else {
        double b[2] = {0.0, 0.0};
#pragma unroll 2
        for (int q = 0; q < lim; ++q) {
          const double hx = s_h[q].x, hy = s_h[q].y, hz = s_h[q].z, hm = s_h[q].w;
#pragma unroll
          for (int t = 0; t < 2; ++t) {
            const double dx = X[t] - hx, dy = Y[t] - hy, dz = Z[t] - hz;
            const double r2 = __fma_rn(dx, dx, __fma_rn(dy, dy, dz * dz));
            const RsqrtSeed u = rsqrt_seed(r2);
            double ir = __fma_rn(u.y * u.e, __fma_rn(0.375, u.e, 0.5), u.y);
            // two bodies at one place: infinite, as 1 / r; the target itself: none
            if (__double_as_longlong(r2) == 0)
              ir = J == row && q == t * kEThreads + tid
                       ? 0.0 : __longlong_as_double(0x7ff0000000000000LL);
            b[t] = __fma_rn(hm, ir, b[t]);
          }
        }
        const double w = J == row ? 0.5 : 1.0;
        sd[0] += w * b[0];
        sd[1] += w * b[1];
      }
    }
#pragma unroll
    for (int t = 0; t < 2; ++t)
      if ((int64_t)row * kETile + t * kEThreads + tid < n)
        ep -= prm.G * M[t] * (MIXED ? (double)sh[t] + (double)sl[t] : sd[t]);
    if (rowA == rowB) break;
  }
  double v[3] = {ek, es, ep};
  for (int q = 0; q < 3; ++q)
    for (int o = 16; o > 0; o >>= 1) v[q] += __shfl_xor_sync(0xffffffffu, v[q], o);
  if ((tid & 31) == 0)
    for (int q = 0; q < 3; ++q) s_red[q][tid >> 5] = v[q];
  __syncthreads();
  if (tid < 3) {  // per-block partials, added in block order afterwards
    double s = 0.0;
    for (int w = 0; w < kEThreads / 32; ++w) s += s_red[tid][w];
    part[3 * ((int64_t)blockIdx.y * gridDim.x + blockIdx.x) + tid] = s;
  }
}

// the three sums over the block partials (eight warps each, a fixed strided
// order and shuffle tree): the same result on every run
__global__ void k_energy_final(const double *part, int64_t nblocks, double *out) {
  pdl_wait();
  const int q = threadIdx.x >> 8, t = threadIdx.x & 255, lane = threadIdx.x & 31;
  __shared__ double sum[3][8];
  double s = 0.0;
  for (int64_t b = t; b < nblocks; b += 256) s += part[3 * b + q];
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if (lane == 0) sum[q][t >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    double e[3];
    for (int k = 0; k < 3; ++k) {
      e[k] = 0.0;
      for (int w = 0; w < 8; ++w) e[k] += sum[k][w];
    }
    out[1] = e[0]; out[2] = e[1]; out[3] = e[2];
    out[0] = e[0] + e[1] + e[2];
  }
}


// ---- the merge after the second kick (procedure step 9) --------------------
// One block: every composite's lowest member gets the summed mass and the
// radius of the summed volume; the dissipation totals are summed in a fixed
// order (clusters by label, composites by lowest member) so that they do not
// depend on the order the hard step appended them in.
__global__ void k_merge_sets(const int4 *ent, int64_t ne, const int4 *rec, const double *rec_e,
                             int64_t nrec, const double *esoft, double *m, double *rp,
                             double *sorted_h, double *sorted_s, double *out) {
  pdl_wait();
  for (int64_t s = threadIdx.x; s < ne; s += blockDim.x) {
    const int4 e = ent[s];
    if (e.x != e.y) continue;
    double M = 0.0, V = 0.0;
    for (int l = e.z; l < e.w; ++l) {
      const int q = ent[l].x;
      M += m[q];
      if (rp) V += rp[q] * rp[q] * rp[q];
    }
    m[e.x] = M;
    if (rp) rp[e.x] = cbrt(V);
    int64_t rank = 0;
    for (int64_t u = 0; u < ne; ++u) rank += ent[u].x == ent[u].y && ent[u].y < e.y;
    sorted_s[rank] = esoft[s];
  }
  for (int64_t r = threadIdx.x; r < nrec; r += blockDim.x) {
    int64_t rank = 0;
    for (int64_t u = 0; u < nrec; ++u) rank += rec[u].x < rec[r].x;
    sorted_h[rank] = rec_e[r];
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    int64_t nsets = 0;
    for (int64_t u = 0; u < ne; ++u) nsets += ent[u].x == ent[u].y;
    double eh = 0.0, es = 0.0;
    for (int64_t r = 0; r < nrec; ++r) eh += sorted_h[r];
    for (int64_t q = 0; q < nsets; ++q) es += sorted_s[q];
    out[0] = eh;
    out[1] = es;
  }
}

__global__ void k_merge_keep(int64_t n, const int32_t *slot, const int4 *ent, int32_t *keep) {
  pdl_wait();
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    const int32_t s = slot[i];
    keep[i] = (s < 0 || ent[s].x == ent[s].y) ? 1 : 0;
  }
}

// survivors to their new places in the scratch arrays (10 arrays of n)
__global__ void k_merge_gather(int64_t n, const int32_t *keep, const int64_t *pos,
                               p3t_particles p, double *scr, int32_t *new_index) {
  pdl_wait();
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    if (!keep[i]) {
      new_index[i] = -1;
      continue;
    }
    const int64_t d = pos[i];
    new_index[i] = (int32_t)d;
    scr[d] = p.x[i]; scr[n + d] = p.y[i]; scr[2 * n + d] = p.z[i];
    scr[3 * n + d] = p.vx[i]; scr[4 * n + d] = p.vy[i]; scr[5 * n + d] = p.vz[i];
    scr[6 * n + d] = p.m[i]; scr[7 * n + d] = p.r_out[i]; scr[8 * n + d] = p.r_search[i];
    if (p.r_phys) scr[9 * n + d] = p.r_phys[i];
  }
}

__global__ void k_merge_reset(const int4 *ent, int64_t ne, int32_t *slot,
                              unsigned long long *ctr) {
  pdl_wait();
  for (int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; s < ne;
       s += (int64_t)gridDim.x * blockDim.x)
    slot[ent[s].x] = -1;
  if (blockIdx.x == 0 && threadIdx.x == 0) *ctr = 0ull;
}

__global__ void k_iota(int64_t n, int32_t *a) {
  pdl_wait();
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x)
    a[i] = (int32_t)i;
}

CollOut coll_out(p3t_ctx *c) {
  CollOut co;
  co.ctr = c->coll_ctr;
  co.ent = c->coll_ent;
  co.rec = c->coll_rec;
  co.rec_e = c->coll_rec_e;
  co.slot = c->coll_slot;
  co.ent_cap = c->cap;
  co.rec_cap = c->cap / 2 + 1;
  return co;
}

}  // namespace

int p3t_run_kick(p3t_ctx *c, p3t_particles *p, const double *ax,
                 const double *ay, const double *az, double h, cudaStream_t s) {
  if (p->n == 0) return P3T_OK;
  const int64_t g = p3t_grid(p->n, kBlock, (int64_t)c->num_sms * P3T_NSM_BLOCKS);
  const bool coll = c->prm.f_radius > 0.0;
  pdl_launch(k_kick, dim3((unsigned)g), dim3(kBlock), 0, s, p->n, p->vx, p->vy, p->vz, ax, ay, az, h,
                                        coll ? c->coll_slot : nullptr, c->coll_ent, p->m,
                                        c->coll_esoft);
  p3t_note_launches(1);
  return cudaGetLastError() == cudaSuccess ? P3T_OK : P3T_ERR_CUDA;
}

int p3t_run_hard_step(p3t_ctx *c, p3t_particles *p, const p3t_clusters *cl,
                      double dt, uint64_t *n_steps, cudaStream_t s) {
  const int64_t n = p->n;
  const int64_t maxb = (int64_t)c->num_sms * P3T_NSM_BLOCKS;
  const double mu = c->prm.G * c->prm.m_star;
  HBig big{c->hw, c->ht, c->hl, c->cap};
  const CollOut co = coll_out(c);
  unsigned long long *steps = n_steps ? reinterpret_cast<unsigned long long *>(n_steps)
                                      : c->hsteps;
  pdl_launch(k_zero_hard, dim3(1), dim3(32), 0, s, steps, c->hcursor);
  // the clusters of the four-warp and workspace kernels, listed once so that
  // those kernels do not step through every small cluster
  const int hw = c->hwarp_max;
  pdl_launch(k_cluster_classes, dim3((unsigned)p3t_grid(n / 2 + 1, kBlock, maxb)), dim3(kBlock), 0,
             s, &cl->counts[1], cl->cl_off, hw, c->hlist_cap, c->hlist, c->hcursor + 3);
  // Kepler drift, small clusters and large clusters touch disjoint particles:
  // run them on three streams forked from and joined back to the caller's
  P3T_CUDA_TRY(cudaEventRecord(c->ev_fork, s));
  P3T_CUDA_TRY(cudaStreamWaitEvent(c->aux[0], c->ev_fork, 0));
  P3T_CUDA_TRY(cudaStreamWaitEvent(c->aux[1], c->ev_fork, 0));
  const int64_t ncl_max = (n / 2) > 0 ? n / 2 : 1;
  const HConst hc = hermite_const(c->prm, dt);
  const int64_t nbig = c->num_sms < 32 ? c->num_sms : 32;
  // clusters of 2..hw members: a warp each (stream aux[0]), up to 32 such
  // one-warp blocks an SM (the FP64 latency of their block steps, not the
  // FP64 pipe, limits them: 16 an SM took 40 us more a step); up to 128: a
  // 128-thread block each, then > 128 (stream aux[1])
  const unsigned gw = (unsigned)p3t_grid(ncl_max * 32, 32, (int64_t)c->num_sms * 32);
  if (hw <= 8)
    pdl_launch(k_hermite_block<32, 8, false>, dim3(gw), dim3(32), sizeof(HSmall<8>), c->aux[0], 
        &cl->counts[1], cl->cl_off, cl->cl_mem, *p, c->prm, hc, dt, 2, hw, steps, c->hcursor,
        (const int32_t *)nullptr, (const int64_t *)nullptr, big, co, c->status, c->hermite_limit,
        c->hermite_rec);
  else if (hw <= 16)
    pdl_launch(k_hermite_block<32, 16, false>, dim3(gw), dim3(32), sizeof(HSmall<16>), c->aux[0], 
        &cl->counts[1], cl->cl_off, cl->cl_mem, *p, c->prm, hc, dt, 2, hw, steps, c->hcursor,
        (const int32_t *)nullptr, (const int64_t *)nullptr, big, co, c->status, c->hermite_limit,
        c->hermite_rec);
  else
    pdl_launch(k_hermite_block<32, 32, false>, dim3(gw), dim3(32), sizeof(HSmall<32>), c->aux[0], 
        &cl->counts[1], cl->cl_off, cl->cl_mem, *p, c->prm, hc, dt, 2, hw, steps, c->hcursor,
        (const int32_t *)nullptr, (const int64_t *)nullptr, big, co, c->status, c->hermite_limit,
        c->hermite_rec);
  pdl_launch(k_hermite_block<128, kHMax, false>, dim3((unsigned)p3t_grid(ncl_max * 128, 128, (int64_t)c->num_sms * 2)), dim3(128), sizeof(HSmall<kHMax>), c->aux[1], 
      &cl->counts[1], cl->cl_off, cl->cl_mem, *p, c->prm, hc, dt, hw + 1, kHMax, steps,
      c->hcursor + 1, (const int32_t *)c->hlist, (const int64_t *)(c->hcursor + 3),
      big, co, c->status, c->hermite_limit, c->hermite_rec);
  pdl_launch(k_hermite_block<128, 1, true>, dim3((unsigned)p3t_grid(ncl_max, 1, nbig)), dim3(128), 0, c->aux[1], 
      &cl->counts[1], cl->cl_off, cl->cl_mem, *p, c->prm, hc, dt, kHMax + 1, 0x7fffffff, steps,
      c->hcursor + 2, (const int32_t *)(c->hlist + c->hlist_cap),
      (const int64_t *)(c->hcursor + 4), big, co, c->status, c->hermite_limit, c->hermite_rec);
  KepConst kc;
  kc.mu = mu;
  kc.sq = sqrt(mu);
  kc.isq = 1.0 / kc.sq;
  kc.imu = 1.0 / mu;
  auto kep = c->prm.precision == P3T_MIXED ? k_kepler<true> : k_kepler<false>;
  pdl_launch(kep, dim3((unsigned)p3t_grid(n, 128, maxb)), dim3(128), 0, s, &cl->counts[0], cl->singles, *p, dt, kc,
                                                        c->status);
  P3T_CUDA_TRY(cudaEventRecord(c->ev_join[0], c->aux[0]));
  P3T_CUDA_TRY(cudaEventRecord(c->ev_join[1], c->aux[1]));
  P3T_CUDA_TRY(cudaStreamWaitEvent(s, c->ev_join[0], 0));
  P3T_CUDA_TRY(cudaStreamWaitEvent(s, c->ev_join[1], 0));
  p3t_note_launches(6);
  return cudaGetLastError() == cudaSuccess ? P3T_OK : P3T_ERR_CUDA;
}

int p3t_run_kepler_drift(p3t_ctx *c, p3t_particles *p, double dt, cudaStream_t s) {
  if (p->n == 0) return P3T_OK;
  KepConst kc;
  kc.mu = c->prm.G * c->prm.m_star;
  kc.sq = sqrt(kc.mu);
  kc.isq = 1.0 / kc.sq;
  kc.imu = 1.0 / kc.mu;
  auto kep = c->prm.precision == P3T_MIXED ? k_kepler_all<true> : k_kepler_all<false>;
  pdl_launch(kep, dim3((unsigned)p3t_grid(p->n, 128, (int64_t)c->num_sms * P3T_NSM_BLOCKS)), dim3(128), 0, s, 
      *p, dt, kc, c->status);
  p3t_note_launches(1);
  return cudaGetLastError() == cudaSuccess ? P3T_OK : P3T_ERR_CUDA;
}

// Procedure step 9 for composites (Sec. 2.4.1).  Synchronises the stream: the
// caller needs the new particle count on the host.
int p3t_run_merge(p3t_ctx *c, p3t_particles *p, int32_t *new_index, double *e_disp,
                  int64_t *n_merged, cudaStream_t s) {
  const int64_t n = p->n;
  const int64_t maxb = (int64_t)c->num_sms * P3T_NSM_BLOCKS;
  unsigned long long ctr = 0;
  P3T_CUDA_TRY(cudaMemcpyAsync(&ctr, c->coll_ctr, sizeof(ctr), cudaMemcpyDeviceToHost, s));
  P3T_CUDA_TRY(cudaStreamSynchronize(s));
  int64_t nrec = (int64_t)(ctr >> 32), ne = (int64_t)(ctr & 0xffffffffull);
  const CollOut co = coll_out(c);
  if (nrec > co.rec_cap) nrec = co.rec_cap;  // a capacity error is already recorded
  if (ne > co.ent_cap) ne = co.ent_cap;
  if (nrec == 0 || ne == 0 || n == 0) {
    if (e_disp) e_disp[0] = e_disp[1] = 0.0;
    if (n_merged) *n_merged = 0;
    if (new_index && n > 0) {
      pdl_launch(k_iota, dim3((unsigned)p3t_grid(n, kBlock, maxb)), dim3(kBlock), 0, s, n, new_index);
      p3t_note_launches(1);
    }
    return cudaGetLastError() == cudaSuccess ? P3T_OK : P3T_ERR_CUDA;
  }
  double *scr = c->hw;              // 10 n for the gather
  double *sorted_h = c->hw + 10 * c->cap, *sorted_s = sorted_h + c->cap;
  double *out = c->epart;
  int32_t *keep = c->flag;
  int64_t *pos = c->pos;
  int32_t *ni = new_index ? new_index : c->flag + c->cap;
  int64_t *d_n = c->counters + 16, *d_total = c->counters + 17;
  P3T_CUDA_TRY(cudaMemcpyAsync(d_n, &n, sizeof(n), cudaMemcpyHostToDevice, s));
  pdl_launch(k_merge_sets, dim3(1), dim3(1024), 0, s, co.ent, ne, co.rec, co.rec_e, nrec, c->coll_esoft, p->m,
                                  p->r_phys, sorted_h, sorted_s, out);
  const unsigned g = (unsigned)p3t_grid(n, kBlock, maxb);
  pdl_launch(k_merge_keep, dim3(g), dim3(kBlock), 0, s, n, c->coll_slot, co.ent, keep);
  int rc = p3t_scan_i32_to_i64(keep, pos, d_n, n, d_total, c->scan_state, c->scan_words, c->status, c->poll_limit, s);
  if (rc) return rc;
  pdl_launch(k_merge_gather, dim3(g), dim3(kBlock), 0, s, n, keep, pos, *p, scr, ni);
  double *dst[10] = {p->x, p->y, p->z, p->vx, p->vy, p->vz, p->m, p->r_out, p->r_search,
                     p->r_phys};
  for (int q = 0; q < 10; ++q)
    if (dst[q])
      P3T_CUDA_TRY(cudaMemcpyAsync(dst[q], scr + q * n, sizeof(double) * n,
                                   cudaMemcpyDeviceToDevice, s));
  pdl_launch(k_merge_reset, dim3((unsigned)p3t_grid(ne, kBlock, maxb)), dim3(kBlock), 0, s, co.ent, ne, c->coll_slot,
                                                                        c->coll_ctr);
  p3t_note_launches(5);
  double eo[2];
  int64_t total = 0;
  P3T_CUDA_TRY(cudaMemcpyAsync(eo, out, sizeof(eo), cudaMemcpyDeviceToHost, s));
  P3T_CUDA_TRY(cudaMemcpyAsync(&total, d_total, sizeof(total), cudaMemcpyDeviceToHost, s));
  P3T_CUDA_TRY(cudaStreamSynchronize(s));
  if (e_disp) { e_disp[0] = eo[0]; e_disp[1] = eo[1]; }
  if (n_merged) *n_merged = n - total;
  p->n = total;
  return cudaGetLastError() == cudaSuccess ? P3T_OK : P3T_ERR_CUDA;
}

int p3t_run_energy(p3t_ctx *c, const p3t_particles *p, double *out, cudaStream_t s) {
  const int64_t tiles = (p->n + kETile - 1) / kETile;
  const int64_t rows = (tiles + 1) / 2;  // folded: T + 1 tile pairs each
  // chunks of tile pairs so that about kEBlocks blocks have one each; the
  // partials, 3 rows ceil((T + 1) / chunk), fit the workspace of 33 cap doubles
  int64_t chunk = rows * (tiles + 1) / kEBlocks;
  if (chunk < 1) chunk = 1;
  const int64_t ny = (tiles + 1 + chunk - 1) / chunk, g = rows * ny;
  double *part = c->hw;
  if (3 * g > 33 * c->cap) return P3T_ERR_CAPACITY;
  if (p->n > 0) {
    auto k = c->prm.precision == P3T_MIXED ? k_energy<true> : k_energy<false>;
    pdl_launch(k, dim3((unsigned)rows, (unsigned)ny), dim3(kEThreads), 0, s, *p, c->prm,
               (int)tiles, (int)chunk, part);
  }
  pdl_launch(k_energy_final, dim3(1), dim3(768), 0, s, part, p->n > 0 ? g : (int64_t)0, out);
  p3t_note_launches(p->n > 0 ? 2 : 1);
  return cudaGetLastError() == cudaSuccess ? P3T_OK : P3T_ERR_CUDA;
}
