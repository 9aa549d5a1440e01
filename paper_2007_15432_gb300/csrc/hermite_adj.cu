// Adjoint of the hard part of a soft step (procedure step 5) for the members
// of neighbour clusters: the vector-Jacobian product of the cluster's
// Hermite-4 block-step integration over [0, dt] (Sec. 2.1.2; Eq. hardforce)
// with the block schedule held fixed, through forward-mode tangents.
//
// A direction is one of a member's six state components or its mass.  Clusters
// of up to kLanesMax members have their components in the lanes of a warp
// (k_tangent_lanes below); larger ones take one thread per (member, direction),
// which integrates the whole cluster in plain FP64 arithmetic (each formula as written: the
// predictor to the jerk, the Makino & Aarseth corrector, the Aarseth step,
// the first step eta0 |a| / |j|, block steps dt / 2^k, k <= 40, at most
// twice the previous one and commensurate with the particle time) carrying
// one tangent along with every value; the step decisions use the values
// only, so the tangent is the derivative of the integration with its
// schedule fixed.  The tangent of the final state, dotted with the adjoint
// of the final state, is one component of Phi^T lam (or dL/dm for a mass
// direction).  Clusters above kTMax members are not integrated here
// (P3T_ERR_CAPACITY).  No collisions (f_radius = 0).
#include <math.h>

#include "hermite_lanes.cuh"
#include "p3t_internal.cuh"

namespace {

constexpr int kTMax = 16;  // largest cluster the tangent kernel integrates
constexpr int kLv = 40;    // finest block level, dt / 2^40

struct D1 {
  double v, d;  // value and tangent
};
__device__ __forceinline__ D1 dk(double v) { return {v, 0.0}; }
__device__ __forceinline__ D1 operator+(D1 a, D1 b) { return {a.v + b.v, a.d + b.d}; }
__device__ __forceinline__ D1 operator-(D1 a, D1 b) { return {a.v - b.v, a.d - b.d}; }
__device__ __forceinline__ D1 operator-(D1 a) { return {-a.v, -a.d}; }
__device__ __forceinline__ D1 operator*(D1 a, D1 b) { return {a.v * b.v, a.d * b.v + a.v * b.d}; }
__device__ __forceinline__ D1 operator*(double s, D1 a) { return {s * a.v, s * a.d}; }
__device__ __forceinline__ D1 operator/(D1 a, D1 b) {
  const double q = a.v / b.v;
  return {q, (a.d - q * b.d) / b.v};
}
__device__ __forceinline__ D1 operator/(D1 a, double s) { return {a.v / s, a.d / s}; }
__device__ __forceinline__ D1 dsqrt(D1 a) {
  const double r = sqrt(a.v);
  return {r, a.v > 0.0 ? a.d / (2.0 * r) : 0.0};
}

// level of the step dt_des: the largest dt / 2^l not above it, l <= 40, at
// most twice the previous step, commensurate with the time t (units dt/2^40)
__device__ int level_of(double dt_des, double dt, int prev, int64_t t, bool &uf) {
  int l = 0;
  while (l < kLv && ldexp(dt, -l) > dt_des) ++l;
  if (ldexp(dt, -l) > dt_des) uf = true;
  if (l < prev - 1) l = prev - 1;
  while (l < kLv && (t & ((((int64_t)1) << (kLv - l)) - 1)) != 0) ++l;
  return l;
}

// hard acceleration and jerk of member k (Eq. hardforce): the star and the
// (1 - K) part of every other member's pull, the jerk with dK/dt
__device__ void acc_jerk(int nc, const D1 (*x)[3], const D1 (*v)[3], const D1 *m,
                         const double *ro, int k, const p3t_params &prm, D1 a[3], D1 j[3]) {
  for (int c = 0; c < 3; ++c) { a[c] = dk(0.0); j[c] = dk(0.0); }
  {
    const D1 r2 = x[k][0] * x[k][0] + x[k][1] * x[k][1] + x[k][2] * x[k][2];
    const D1 r = dsqrt(r2);
    const D1 r3 = r2 * r, r5 = r3 * r2;
    const D1 rv = x[k][0] * v[k][0] + x[k][1] * v[k][1] + x[k][2] * v[k][2];
    const double GM = prm.G * prm.m_star;
    for (int c = 0; c < 3; ++c) {
      a[c] = a[c] - (GM * x[k][c]) / r3;
      j[c] = j[c] - GM * (v[k][c] / r3 - ((3.0 * rv) * x[k][c]) / r5);
    }
  }
  const double i1mg = 1.0 / (1.0 - prm.gamma);
  for (int q = 0; q < nc; ++q) {
    if (q == k) continue;
    D1 rr[3], uu[3];
    for (int c = 0; c < 3; ++c) { rr[c] = x[k][c] - x[q][c]; uu[c] = v[k][c] - v[q][c]; }
    const D1 r2 = rr[0] * rr[0] + rr[1] * rr[1] + rr[2] * rr[2];
    if (r2.v == 0.0) continue;
    const D1 r = dsqrt(r2);
    const double roij = ro[k] > ro[q] ? ro[k] : ro[q];
    const D1 y = r / roij;
    if (y.v >= 1.0) continue;
    D1 w = dk(1.0), dK = dk(0.0);
    if (y.v > prm.gamma) {
      const D1 xs = (y - dk(prm.gamma)) * dk(i1mg);
      const D1 x2 = xs * xs, x3 = x2 * xs, us = dk(1.0) - xs;
      w = dk(1.0) - x2 * x2 * (dk(35.0) - 84.0 * xs + 70.0 * x2 - 20.0 * x3);
      dK = (140.0 * xs * xs * xs * us * us * us) / (1.0 - prm.gamma);
    }
    const D1 r3 = r2 * r, r5 = r3 * r2;
    const D1 rv = rr[0] * uu[0] + rr[1] * uu[1] + rr[2] * uu[2];
    const D1 Gm = prm.G * m[q];
    const D1 dw = dK * rv / (r * dk(roij));  // -d(1 - K)/dt
    for (int c = 0; c < 3; ++c) {
      a[c] = a[c] - Gm * w * rr[c] / r3;
      j[c] = j[c] - Gm * (w * (uu[c] / r3 - ((3.0 * rv) * rr[c]) / r5) - dw * rr[c] / r3);
    }
  }
}

__device__ __forceinline__ double norm3v(const D1 *u) {
  return sqrt(u[0].v * u[0].v + u[1].v * u[1].v + u[2].v * u[2].v);
}

// thread t: member slot u = t / 7 of the cluster list, direction t % 7
// (x, y, z, vx, vy, vz, m); writes the state directions' results to
// lin[6 u + dir] and adds the mass direction's to gm
__global__ void k_hermite_tangent(const int64_t *counts, const int64_t *cl_off,
                                  const int32_t *cl_mem, p3t_particles p, p3t_params prm,
                                  double dt, int nc_min, const double *lx, const double *ly,
                                  const double *lz, const double *lvx, const double *lvy,
                                  const double *lvz, double *lin, double *gm, DevStatus *st) {
  pdl_wait();
  const int64_t ncl = counts[1], nmem = counts[2];
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < 7 * nmem;
       t += (int64_t)gridDim.x * blockDim.x) {
    const int64_t u = t / 7;
    const int dir = (int)(t - 7 * u);
    int64_t lo = 0, hi = ncl;  // the cluster c with cl_off[c] <= u < cl_off[c + 1]
    while (hi - lo > 1) {
      const int64_t mid = (lo + hi) / 2;
      if (cl_off[mid] <= u) lo = mid; else hi = mid;
    }
    const int64_t off = cl_off[lo];
    const int nc = (int)(cl_off[lo + 1] - off);
    if (nc > kTMax) {
      dev_fail(st, P3T_ERR_CAPACITY, 80, nc);
      continue;
    }
    if (nc < nc_min) continue;  // k_tangent_lanes'
    const int ks = (int)(u - off);  // the seeded member
    D1 x[kTMax][3], v[kTMax][3], a[kTMax][3], jk[kTMax][3], m[kTMax];
    D1 px[kTMax][3], pv[kTMax][3], a1[kTMax][3], j1[kTMax][3];
    double ro[kTMax];
    int64_t tt[kTMax];
    int lvl[kTMax];
    bool act[kTMax];
    for (int k = 0; k < nc; ++k) {
      const int32_t i = cl_mem[off + k];
      x[k][0] = dk(p.x[i]); x[k][1] = dk(p.y[i]); x[k][2] = dk(p.z[i]);
      v[k][0] = dk(p.vx[i]); v[k][1] = dk(p.vy[i]); v[k][2] = dk(p.vz[i]);
      m[k] = dk(p.m[i]);
      ro[k] = p.r_out[i];
    }
    if (dir < 3) x[ks][dir].d = 1.0;
    else if (dir < 6) v[ks][dir - 3].d = 1.0;
    else m[ks].d = 1.0;
    const int64_t T = ((int64_t)1) << kLv;
    const double unit = ldexp(dt, -kLv);
    bool uf = false;
    for (int k = 0; k < nc; ++k) {
      acc_jerk(nc, x, v, m, ro, k, prm, a[k], jk[k]);
      const double jn = norm3v(jk[k]);
      const double d0 = jn > 0.0 ? prm.eta0 * norm3v(a[k]) / jn : dt;
      tt[k] = 0;
      lvl[k] = level_of(d0, dt, 0, 0, uf);
    }
    for (int64_t blocks = 0; !uf; ++blocks) {
      if (blocks > ((int64_t)1 << 24)) { dev_fail(st, P3T_ERR_TIMEOUT, 81, 0); break; }
      int64_t tn = T, tmin = T;
      for (int k = 0; k < nc; ++k) {
        const int64_t e = tt[k] + (T >> lvl[k]);
        tn = e < tn ? e : tn;
        tmin = tt[k] < tmin ? tt[k] : tmin;
      }
      if (tmin >= T) break;
      for (int k = 0; k < nc; ++k) {
        const double D = (double)(tn - tt[k]) * unit, D2 = D * D, D3 = D2 * D;
        for (int c = 0; c < 3; ++c) {
          px[k][c] = x[k][c] + D * v[k][c] + (D2 * a[k][c]) / 2.0 + (D3 * jk[k][c]) / 6.0;
          pv[k][c] = v[k][c] + D * a[k][c] + (D2 * jk[k][c]) / 2.0;
        }
        act[k] = tt[k] + (T >> lvl[k]) == tn;
      }
      for (int k = 0; k < nc; ++k)
        if (act[k]) acc_jerk(nc, px, pv, m, ro, k, prm, a1[k], j1[k]);
      for (int k = 0; k < nc; ++k) {
        if (!act[k]) continue;
        const double D = (double)(T >> lvl[k]) * unit;
        const double D2 = D * D, D3 = D2 * D, D4 = D3 * D, D5 = D4 * D;
        D1 A2[3], A3[3], A2e[3];
        for (int c = 0; c < 3; ++c) {
          const D1 da = a[k][c] - a1[k][c];
          A2[c] = (-6.0 * da - D * (4.0 * jk[k][c] + 2.0 * j1[k][c])) / D2;
          A3[c] = (12.0 * da + (6.0 * D) * (jk[k][c] + j1[k][c])) / D3;
          A2e[c] = A2[c] + D * A3[c];
        }
        for (int c = 0; c < 3; ++c) {
          x[k][c] = px[k][c] + (D4 * A2[c]) / 24.0 + (D5 * A3[c]) / 120.0;
          v[k][c] = pv[k][c] + (D3 * A2[c]) / 6.0 + (D4 * A3[c]) / 24.0;
          a[k][c] = a1[k][c];
          jk[k][c] = j1[k][c];
        }
        const double an = norm3v(a[k]), jn = norm3v(jk[k]);
        const double a2n = norm3v(A2e), a3n = norm3v(A3);
        const double num = an * a2n + jn * jn, den = jn * a3n + a2n * a2n;
        const double dd = den > 0.0 ? sqrt(prm.eta * num / den) : dt;
        tt[k] = tn;
        lvl[k] = level_of(dd, dt, lvl[k], tn, uf);
      }
    }
    if (uf) dev_fail(st, P3T_ERR_DT_UNDERFLOW, 82, 0);
    double r = 0.0;
    for (int k = 0; k < nc; ++k) {
      const int32_t i = cl_mem[off + k];
      r += lx[i] * x[k][0].d + ly[i] * x[k][1].d + lz[i] * x[k][2].d +
           lvx[i] * v[k][0].d + lvy[i] * v[k][1].d + lvz[i] * v[k][2].d;
    }
    if (dir < 6) lin[6 * u + dir] = r;
    else gm[cl_mem[u]] += r;
  }
}

// ---- clusters of at most ten members: a lane per member component --------------
// A warp carries up to 32 / (3 nc) directions of one member, each in 3 nc lanes
// (member k, component c: value and tangent of x, v, a, j in registers); dot
// products are taken over a member's three lanes by shuffles.  The directions
// of a warp share the values, so the block schedule is the same in all of its
// lanes.  What bounds it is the latency of one cluster's block steps, each FP64
// warp instruction 64 cycles: the formulas are written for few of them (powers
// of 1 / r from one seed, no division, differentiated by hand: with s = r.dr, h
// = s / r^2, d r^-2 = -2 h r^-2, d r^-3 = -3 h r^-3), about 42 for the star, 52
// for a pair inside gamma r_out and 92 in the changeover, 45 for predictor and
// corrector, where a thread per direction in dual numbers took some 2,000 a
// block step of a pair.  Measured: N = 10,000 ring, 1,524 -> 137 us a call.
struct TanOut {
  double a, j, da, dj;
};

// step criterion as k_hermite_tangent evaluates it, from the members' own
// components (three lanes from b0 on)
__device__ __noinline__ double exact_step64(double a, double j, double a2, double a3, int b0,
                                            bool later, double eta, double eta0, double dt) {
  double n[4];
  const double u[4] = {a, j, a2, a3};
  for (int q = 0; q < 4; ++q) {
    const double s = u[q] * u[q];
    n[q] = sqrt(shfl_d(s, b0 & 31) + shfl_d(s, (b0 + 1) & 31) + shfl_d(s, (b0 + 2) & 31));
  }
  if (!later) return n[1] > 0.0 ? eta0 * n[0] / n[1] : dt;
  const double num = n[0] * n[2] + n[1] * n[1], den = n[1] * n[3] + n[2] * n[2];
  return den > 0.0 ? sqrt(eta * num / den) : dt;
}

// a member's three components of v, from its lanes
__device__ __forceinline__ void row3(double v, int b0, double (&o)[3]) {
  o[0] = shfl_d(v, b0 & 31);
  o[1] = shfl_d(v, (b0 + 1) & 31);
  o[2] = shfl_d(v, (b0 + 2) & 31);
}
__device__ __forceinline__ double dot3(const double (&a)[3], const double (&b)[3]) {
  return __fma_rn(a[0], b[0], __fma_rn(a[1], b[1], a[2] * b[2]));
}

// hard acceleration and jerk of the lane's member and component, with their
// tangents, from every member's (p, v, dp, dv) in the lanes
__device__ __forceinline__ TanOut hard_tangent(int nc, int k, int b0, int row0, double p, double v,
                                               double dp, double dv, double gm, double dgm,
                                               double iro, const p3t_params &prm,
                                               const HConst &hc) {
  TanOut o;
  {  // the star
    double r[3], u[3], dr[3], du[3];
    row3(p, b0, r);
    row3(v, b0, u);
    row3(dp, b0, dr);
    row3(dv, b0, du);
    const double r2 = dot3(r, r), s = dot3(r, dr), rv = dot3(r, u);
    const double drv = dot3(dr, u) + dot3(r, du);
    const RsqrtSeed i = rsqrt_seed(r2);
    const double y = i.y, y2 = i.y2, e = i.e, y3 = y2 * y;
    const double ri3 = __fma_rn(y3 * e, __fma_rn(1.875, e, 1.5), y3);
    const double ri2 = __fma_rn(y2, __fma_rn(e, e, e), y2);
    const double g = -hc.gms * ri3, h = ri2 * s, r3i2 = 3.0 * ri2;
    const double al = r3i2 * rv, dg = -3.0 * g * h;
    const double dal = __fma_rn(r3i2, drv, -2.0 * (al * h));
    const double t = __fma_rn(-al, p, v);
    const double dt = __fma_rn(-dal, p, __fma_rn(-al, dp, dv));
    o.a = g * p;
    o.j = g * t;
    o.da = __fma_rn(dg, p, g * dp);
    o.dj = __fma_rn(dg, t, g * dt);
  }
  for (int m = 0; m < nc - 1; ++m) {
    const int q = m < k ? m : m + 1;  // the other members by index
    const int src = (row0 + 3 * q + ((threadIdx.x & 31) - b0)) & 31;
    const double rc = p - shfl_d(p, src), uc = v - shfl_d(v, src);
    const double drc = dp - shfl_d(dp, src), duc = dv - shfl_d(dv, src);
    const double G = shfl_d(gm, src), dG = shfl_d(dgm, src), io = shfl_d(iro, src);
    const double irot =
        __double_as_longlong(iro) < __double_as_longlong(io) ? iro : io;  // 1 / max(r_out)
    double r[3], u[3], dr[3], du[3];
    row3(rc, b0, r);
    row3(uc, b0, u);
    row3(drc, b0, dr);
    row3(duc, b0, du);
    const double r2 = dot3(r, r), s = dot3(r, dr), rv = dot3(r, u);
    const double drv = dot3(dr, u) + dot3(r, du);
    const RsqrtSeed i = rsqrt_seed(r2);
    const double y = i.y, y2 = i.y2, e = i.e, y3 = y2 * y;
    const double ri3 = __fma_rn(y3 * e, __fma_rn(1.875, e, 1.5), y3);
    const double ri2 = __fma_rn(y2, __fma_rn(e, e, e), y2);
    const double ri = __fma_rn(y * e, __fma_rn(0.375, e, 0.5), y);
    const double yv = (r2 * ri) * irot;
    // a pair at one place or beyond r_out adds nothing
    const bool off = __double_as_longlong(r2) == 0 || ge_pos(yv, 1.0);
    const bool mid = !off && gt_pos(yv, prm.gamma);
    const double g = off ? 0.0 : -G * ri3, h = ri2 * s, r3i2 = 3.0 * ri2;
    const double al = r3i2 * rv;
    const double dg = off ? 0.0 : __fma_rn(-dG, ri3, -3.0 * g * h);
    const double dal = __fma_rn(r3i2, drv, -2.0 * (al * h));
    double t = __fma_rn(-al, rc, uc);
    double dt = __fma_rn(-dal, rc, __fma_rn(-al, drc, duc));
    double w = rc, dw = drc;  // W r and its tangent
    if (__any_sync(0xffffffffu, mid)) {
      const double xs = (yv - prm.gamma) * hc.i1mg, us = 1.0 - xs;
      const double x2 = xs * xs, u2 = us * us;
      const double K = (x2 * x2) *
                       __fma_rn(__fma_rn(__fma_rn(-20.0, xs, 70.0), xs, -84.0), xs, 35.0);
      const double q2 = (140.0 * hc.i1mg) * (x2 * u2);
      const double W = mid ? 1.0 - K : 1.0;
      const double dK = mid ? q2 * (xs * us) : 0.0;                    // K'(y)
      const double ddK = mid ? (3.0 * hc.i1mg) * (q2 * (us - xs)) : 0.0;  // K''(y)
      // zero outside: irot is infinite between two members of zero radius
      const double rio = mid ? ri * irot : 0.0, dy = s * rio;
      const double dW = -(dK * dy);
      const double ro = rv * rio;
      const double E = dK * ro;  // -dW/dt
      // tangent of E = K' (r.u) / (r r_out)
      const double dE = __fma_rn(ddK * dy, ro, dK * __fma_rn(drv, rio, -(ro * h)));
      dt = __fma_rn(dW, t, __fma_rn(W, dt, -__fma_rn(dE, rc, E * drc)));
      t = __fma_rn(W, t, -(E * rc));
      dw = __fma_rn(dW, rc, W * drc);
      w = W * rc;
    }
    o.a = __fma_rn(g, w, o.a);
    o.j = __fma_rn(g, t, o.j);
    o.da = __fma_rn(dg, w, __fma_rn(g, dw, o.da));
    o.dj = __fma_rn(dg, t, __fma_rn(g, dt, o.dj));
  }
  return o;
}

constexpr int kLanesMax = 10;  // largest cluster whose members' components fit a warp

__global__ void __launch_bounds__(128) k_tangent_lanes(
    const int64_t *counts, const int64_t *cl_off, const int32_t *cl_mem, p3t_particles p,
    p3t_params prm, HConst hc, double dt, const double *lx, const double *ly, const double *lz,
    const double *lvx, const double *lvy, const double *lvz, double *lin, double *gm_out,
    DevStatus *st) {
  pdl_wait();
  const int64_t ncl = counts[1], nmem = counts[2];
  const int lane = threadIdx.x & 31;
  const int64_t T = ((int64_t)1) << kLv;
  const long long bd = __double_as_longlong(dt);
  const int e_unit = ((__double2hiint(hc.unit) >> 20) & 0x7ff) - 1023;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  // unit: slot `part` of the directions of member slot u
  for (int64_t unit = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5; unit < 7 * nmem;
       unit += nw) {
    const int64_t u = unit / 7;
    const int part = (int)(unit - 7 * u);
    int64_t lo = 0, hi = ncl;  // the cluster c with cl_off[c] <= u < cl_off[c + 1]
    while (hi - lo > 1) {
      const int64_t mid = (lo + hi) / 2;
      if (cl_off[mid] <= u) lo = mid; else hi = mid;
    }
    const int64_t off = cl_off[lo];
    const int nc = (int)(cl_off[lo + 1] - off);
    if (nc > kLanesMax) continue;  // k_hermite_tangent's
    const int wid = 3 * nc, per = 32 / wid;  // lanes a direction, directions a warp
    if (part * per >= 7) continue;
    const int dl = lane / wid, rem = lane - dl * wid;
    const int dir = part * per + dl;
    const bool on = dl < per && dir < 7;
    const int k = rem / 3, c = rem - 3 * k;
    const int row0 = lane - rem, b0 = lane - c;
    const int ks = (int)(u - off);  // the seeded member
    const int32_t i = cl_mem[off + k];
    double x = (c == 0 ? p.x : (c == 1 ? p.y : p.z))[i];
    double v = (c == 0 ? p.vx : (c == 1 ? p.vy : p.vz))[i];
    double dx = k == ks && dir == c ? 1.0 : 0.0, dv = k == ks && dir == 3 + c ? 1.0 : 0.0;
    const double gm = prm.G * p.m[i], dgm = k == ks && dir == 6 ? prm.G : 0.0;
    const double iro = 1.0 / p.r_out[i];
    double a = 0.0, j = 0.0, da = 0.0, dj = 0.0;
    double px = x, pv = v, dpx = dx, dpv = dv;
    int64_t t = 0, tn = 0, e_end = 0;
    int lvl = 0;
    bool uf = false;
    for (int64_t blocks = 0;; ++blocks) {
      const bool act = e_end == tn;
      const TanOut f = hard_tangent(nc, k, b0, row0, px, pv, dpx, dpv, gm, dgm, iro, prm, hc);
      double A2 = 0.0, A3 = 0.0, a2e = 0.0;
      int e = e_unit + kLv;
      if (blocks > 0) {
        const int sh = kLv - lvl;
        const double D = shift_exp(hc.unit, sh), mD2 = -shift_exp(hc.unit, sh + 1),
                     D6 = shift_exp(hc.unit6, sh);
        const double iD2 = shift_exp(hc.idt2, 2 * lvl), iD3 = shift_exp(hc.idt3, 3 * lvl);
        const double c3 = shift_exp(hc.c3u, 3 * sh), c4 = shift_exp(hc.c4u, 4 * sh),
                     c5 = shift_exp(hc.c5u, 5 * sh);
        const double d = a - f.a, dd = da - f.da;
        A2 = __fma_rn(mD2, __fma_rn(2.0, j, f.j), -6.0 * d) * iD2;
        A3 = __fma_rn(D6, j + f.j, 12.0 * d) * iD3;
        const double B2 = __fma_rn(mD2, __fma_rn(2.0, dj, f.dj), -6.0 * dd) * iD2;
        const double B3 = __fma_rn(D6, dj + f.dj, 12.0 * dd) * iD3;
        a2e = __fma_rn(D, A3, A2);
        e = e_unit + sh;
        if (act) {
          x = __fma_rn(A3, c5, __fma_rn(A2, c4, px));
          v = __fma_rn(A3, c4, __fma_rn(A2, c3, pv));
          dx = __fma_rn(B3, c5, __fma_rn(B2, c4, dpx));
          dv = __fma_rn(B3, c4, __fma_rn(B2, c3, dpv));
        }
      }
      // the new level: from squared norms of the components' leading 20 bits, by
      // the criterion as written where those do not decide it
      double dtd;
      {
        const float an = norm_lanes(lead_float(f.a, 0), b0), jn = norm_lanes(lead_float(f.j, e), b0);
        const float a2n = norm_lanes(lead_float(a2e, 2 * e), b0),
                    a3n = norm_lanes(lead_float(A3, 3 * e), b0);
        const bool decided = step_estimate(an, jn, a2n, a3n, e, blocks > 0, hc, bd, dtd);
        if (__any_sync(0xffffffffu, on && act && !decided))
          dtd = exact_step64(f.a, f.j, a2e, A3, b0, blocks > 0, prm.eta, prm.eta0, dt);
      }
      if (act) {
        a = f.a;
        j = f.j;
        da = f.da;
        dj = f.dj;
        t = tn;
        lvl = level_bits(dtd, bd, blocks > 0 ? lvl : 0, tn, uf);
      }
      if (__any_sync(0xffffffffu, on && uf)) {
        if (lane == 0) dev_fail(st, P3T_ERR_DT_UNDERFLOW, 82, 0);
        break;
      }
      if (tn >= T) break;
      if (blocks > ((int64_t)1 << 24)) {
        if (lane == 0) dev_fail(st, P3T_ERR_TIMEOUT, 81, 0);
        break;
      }
      e_end = t + (T >> lvl);
      tn = warp_min64(on && e_end < T ? e_end : T);
      // predict, values and tangents (as integrate_five)
      const double D = __fma_rn(__longlong_as_double(0x4330000000000000LL + (tn - t)), hc.unit,
                                hc.m52u);
      const double Dh = shift_exp(D, -1);
      px = __fma_rn(__fma_rn(__fma_rn(j * (1.0 / 3.0), D, a), Dh, v), D, x);
      pv = __fma_rn(__fma_rn(j, Dh, a), D, v);
      dpx = __fma_rn(__fma_rn(__fma_rn(dj * (1.0 / 3.0), D, da), Dh, dv), D, dx);
      dpv = __fma_rn(__fma_rn(dj, Dh, da), D, dv);
    }
    // the final tangent against the final adjoint, the direction's lanes added
    // in lane order
    double r = (c == 0 ? lx : (c == 1 ? ly : lz))[i] * dx +
               (c == 0 ? lvx : (c == 1 ? lvy : lvz))[i] * dv;
    double sum = 0.0;
    for (int q = 0; q < wid; ++q) sum += shfl_d(r, (row0 + q) & 31);
    if (on && rem == 0) {
      if (dir < 6) lin[6 * u + dir] = sum;
      else gm_out[cl_mem[u]] += sum;
    }
    __syncwarp();
  }
}

// the members' adjoints before the hard step, from lin
__global__ void k_member_adjoint(const int64_t *counts, const int32_t *cl_mem, const double *lin,
                                 double *lx, double *ly, double *lz, double *lvx, double *lvy,
                                 double *lvz) {
  pdl_wait();
  const int64_t nmem = counts[2];
  for (int64_t u = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; u < nmem;
       u += (int64_t)gridDim.x * blockDim.x) {
    const int32_t i = cl_mem[u];
    lx[i] = lin[6 * u]; ly[i] = lin[6 * u + 1]; lz[i] = lin[6 * u + 2];
    lvx[i] = lin[6 * u + 3]; lvy[i] = lin[6 * u + 4]; lvz[i] = lin[6 * u + 5];
  }
}

}  // namespace

// Phi^T lam for the hard part of a soft step: cluster members through the
// tangent kernel, isolated particles through the Kepler drift's adjoint
// (applied to every particle first; the members' results then replace it)
int p3t_run_hard_step_vjp(p3t_ctx *c, const p3t_particles *p, const p3t_clusters *cl, double dt,
                          double *lx, double *ly, double *lz, double *lvx, double *lvy,
                          double *lvz, double *gm, cudaStream_t s) {
  const int64_t n = p->n;
  if (n == 0) return P3T_OK;
  const int64_t maxb = (int64_t)c->num_sms * P3T_NSM_BLOCKS;
  // clusters of up to ten members by lanes, larger ones (rare) and steps whose
  // scaled constants leave the normal range by a thread per direction
  const HConst hc = hermite_const(c->prm, dt);
  if (hc.fast) {
    pdl_launch(k_tangent_lanes, dim3((unsigned)p3t_grid(7 * n * 32, 128, (int64_t)c->num_sms * 4)),
               dim3(128), 0, s, cl->counts, cl->cl_off, cl->cl_mem, *p, c->prm, hc, dt, lx, ly, lz,
               lvx, lvy, lvz, c->hadj, gm, c->status);
    p3t_note_launches(1);
  }
  pdl_launch(k_hermite_tangent, dim3((unsigned)p3t_grid(7 * n, 128, maxb)), dim3(128), 0, s,
      cl->counts, cl->cl_off, cl->cl_mem, *p, c->prm, dt, hc.fast ? kLanesMax + 1 : 0, lx, ly, lz,
      lvx, lvy, lvz, c->hadj, gm, c->status);
  int rc = p3t_run_kepler_vjp(c, p, dt, lx, ly, lz, lvx, lvy, lvz, s);
  if (rc) return rc;
  pdl_launch(k_member_adjoint, dim3((unsigned)p3t_grid(n, 128, maxb)), dim3(128), 0, s, cl->counts, cl->cl_mem,
                                                                     c->hadj, lx, ly, lz, lvx,
                                                                     lvy, lvz);
  p3t_note_launches(2);
  return cudaGetLastError() == cudaSuccess ? P3T_OK : P3T_ERR_CUDA;
}
