// Adjoint: the vector-Jacobian product of the Kepler drift of every particle
// (the drift of a particle with no neighbours, Sec. 2.1.2) for the adjoint
// of the soft kick-drift-kick (the soft force's VJP is in direct.cu).
//
// The product lam^T Phi is formed in reverse through the drift's formulas, the
// universal anomaly's part from the implicit function theorem (F(chi) = 0
// gives d chi = -dF / F').  What bounds it is the latency of one warp's FP64
// instructions (64 cycles each): some 300 of them, against 1,200 for the
// forward map in dual numbers with six directions.  Measured, N = 1e4:
// 40.8 -> 14.8 us.
#include <math.h>

#include "p3t_internal.cuh"

namespace {

// 1 / n! as a double (exact product of the integers up to 18!, then one
// rounding per factor)
__host__ __device__ constexpr double inv_fact(int n) {
  double f = 1.0;
  for (int i = 2; i <= n; ++i) f *= (double)i;
  return 1.0 / f;
}

// Stumpff functions C(z) = (1 - cos sqrt z) / z, S(z) = (sqrt z - sin sqrt z) /
// z^(3/2) (hyperbolic forms for z < 0) and their derivatives C', S' as plain
// numbers.  |z| < 1: the series C = sum (-z)^k / (2k+2)!, S = sum (-z)^k /
// (2k+3)! and their term-by-term derivatives, NT terms; otherwise the closed
// forms with C' = (1 - z S - 2C) / (2z), S' = (C - 3S) / (2z).
template <int NT>
__device__ __forceinline__ void stumpff_series(double z, double &C, double &S, double &dC,
                                               double &dS) {
  const double mz = -z;
  double c = inv_fact(2 * NT), s_ = inv_fact(2 * NT + 1);
  double dc_ = (double)(NT - 1) * c, ds_ = (double)(NT - 1) * s_;
#pragma unroll
  for (int k = NT - 2; k >= 0; --k) {
    c = fma(mz, c, inv_fact(2 * k + 2));
    s_ = fma(mz, s_, inv_fact(2 * k + 3));
    if (k >= 1) {
      dc_ = fma(mz, dc_, (double)k * inv_fact(2 * k + 2));
      ds_ = fma(mz, ds_, (double)k * inv_fact(2 * k + 3));
    }
  }
  C = c;
  S = s_;
  dC = -dc_;
  dS = -ds_;
}

__device__ void stumpff4(double z, double &C, double &S, double &dC, double &dS) {
  if (fabs(z) < 0.01) {
    stumpff_series<6>(z, C, S, dC, dS);  // truncation below |z|^6 / 14! ~ 1e-23
  } else if (fabs(z) < 1.0) {
    stumpff_series<12>(z, C, S, dC, dS);  // below 1 / 26! ~ 2.5e-27
  } else {
    if (z > 0.0) {
      const double q = sqrt(z);
      C = (1.0 - cos(q)) / z;
      S = (q - sin(q)) / (z * q);
    } else {
      const double q = sqrt(-z);
      C = (cosh(q) - 1.0) / (-z);
      S = (sinh(q) - q) / (-z * q);
    }
    const double i2z = 0.5 / z;
    dC = (1.0 - z * S - 2.0 * C) * i2z;
    dS = (C - 3.0 * S) * i2z;
  }
}

// the universal anomaly (values only), Newton from the series inversion
__device__ double chi_solve(double r0, double sig, double bet, double alpha, double tau,
                            double dt, double mu) {
  const double ir0 = 1.0 / r0, x1 = tau * ir0;
  double chi = x1 * (1.0 - 0.5 * sig * x1 * ir0 +
                     (0.5 * sig * sig * ir0 * ir0 - bet * ir0 / 6.0) * x1 * x1);
  if (alpha > 0.0 && 16.0 * dt * dt * alpha * alpha * alpha * mu > 4.0 * 9.869604401089358)
    chi = tau * alpha;
  for (int it = 0; it < 64; ++it) {
    const double z = alpha * chi * chi, chi2 = chi * chi;
    double C, S, dC, dS;
    stumpff4(z, C, S, dC, dS);
    const double F = sig * chi2 * C + bet * chi2 * chi * S + r0 * chi - tau;
    const double Fp = sig * chi * (1.0 - z * S) + bet * chi2 * C + r0;
    double d = F / Fp;
    const double lim = 0.5 * (fabs(chi) + r0);
    d = d > lim ? lim : (d < -lim ? -lim : d);
    chi -= d;
    if (fabs(d) <= 1e-15 * fabs(chi) || d == 0.0) break;
  }
  return chi;
}

__device__ __forceinline__ double dot3(const double (&a)[3], const double (&b)[3]) {
  return fma(a[0], b[0], fma(a[1], b[1], a[2] * b[2]));
}

// lam_in = Phi^T lam_out for the drift of one particle by dt (sq = sqrt mu, isq
// = 1 / sq, imu = 1 / mu).  With C, S the Stumpff functions at z = alpha chi^2:
// c2 = chi^2 C, c3 = chi^3 S, c1 = (z S - 1) chi; x' = f x + g v and v' = fd x
// + gd v with f = 1 - c2 / r0, g = dt - c3 / sq, fd = sq c1 / (r r0), gd = 1 -
// c2 / r.  A name ending in b is the adjoint of the name before it.
__global__ void k_kepler_vjp(int64_t n, const double *x, const double *y, const double *z,
                             const double *vx, const double *vy, const double *vz, double dt,
                             double mu, double sq, double isq, double imu, double *lx, double *ly,
                             double *lz, double *lvx, double *lvy, double *lvz) {
  pdl_wait();
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    const double X[3] = {x[i], y[i], z[i]}, V[3] = {vx[i], vy[i], vz[i]};
    const double L[3] = {lx[i], ly[i], lz[i]}, Lv[3] = {lvx[i], lvy[i], lvz[i]};
    const double r0 = sqrt(dot3(X, X)), ir0 = 1.0 / r0;
    const double alpha = 2.0 * ir0 - imu * dot3(V, V);
    const double sig = isq * dot3(X, V), bet = 1.0 - alpha * r0;
    const double chi = chi_solve(r0, sig, bet, alpha, sq * dt, dt, mu);
    const double chi2 = chi * chi, chi3 = chi2 * chi, zz = alpha * chi2;
    double C, S, dC, dS;
    stumpff4(zz, C, S, dC, dS);
    const double w = zz * S - 1.0;
    const double c1 = w * chi, c2 = chi2 * C, c3 = chi3 * S;
    const double f = 1.0 - c2 * ir0, g = dt - isq * c3;
    double nx[3];
    for (int a = 0; a < 3; ++a) nx[a] = f * X[a] + g * V[a];
    const double ir = 1.0 / sqrt(dot3(nx, nx)), irr = sq * ir * ir0;
    const double fd = irr * c1, gd = 1.0 - c2 * ir;
    // v'
    const double fdb = dot3(Lv, X), gdb = dot3(Lv, V);
    const double c1b = fdb * irr;
    const double rb = (gdb * c2 * ir - fdb * fd) * ir;
    double r0b = -fdb * fd * ir0;
    // x', with r = |x'|
    const double rbr = rb * ir;
    double nb[3];
    for (int a = 0; a < 3; ++a) nb[a] = L[a] + rbr * nx[a];
    const double fb = dot3(nb, X), gb = dot3(nb, V);
    const double c2b = -gdb * ir - fb * ir0, c3b = -isq * gb;
    r0b += fb * c2 * ir0 * ir0;
    // c1, c2, c3 -> chi, z
    const double zb = c1b * (S * chi + zz * chi * dS) + c3b * chi3 * dS + c2b * chi2 * dC;
    const double chib = c1b * w + 2.0 * c2b * chi * C + 3.0 * c3b * chi2 * S +
                        2.0 * zb * alpha * chi;
    double ab = zb * chi2;
    // chi: F = sig c2 + bet c3 + r0 chi - tau = 0
    const double Fb = -chib / (bet * c2 - sig * c1 + r0);
    ab += Fb * (sig * chi2 * dC + bet * chi3 * dS) * chi2;
    const double rvb = isq * Fb * c2, betb = Fb * c3;
    ab -= betb * r0;
    r0b += Fb * chi - betb * alpha - 2.0 * ab * ir0 * ir0;
    const double vb = -2.0 * imu * ab, xb = r0b * ir0;
    double o[3], ov[3];
    for (int a = 0; a < 3; ++a) {
      o[a] = fd * Lv[a] + f * nb[a] + rvb * V[a] + xb * X[a];
      ov[a] = gd * Lv[a] + g * nb[a] + rvb * X[a] + vb * V[a];
    }
    lx[i] = o[0]; ly[i] = o[1]; lz[i] = o[2];
    lvx[i] = ov[0]; lvy[i] = ov[1]; lvz[i] = ov[2];
  }
}

}  // namespace

int p3t_run_kepler_vjp(p3t_ctx *c, const p3t_particles *p, double dt, double *lx, double *ly,
                       double *lz, double *lvx, double *lvy, double *lvz, cudaStream_t s) {
  const int64_t n = p->n;
  if (n == 0) return P3T_OK;
  const double mu = c->prm.G * c->prm.m_star, sq = sqrt(mu);
  pdl_launch(k_kepler_vjp, dim3((unsigned)p3t_grid(n, 128, (int64_t)c->num_sms * P3T_NSM_BLOCKS)),
             dim3(128), 0, s, n, p->x, p->y, p->z, p->vx, p->vy, p->vz, dt, mu, sq, 1.0 / sq,
             1.0 / mu, lx, ly, lz, lvx, lvy, lvz);
  p3t_note_launches(1);
  return cudaGetLastError() == cudaSuccess ? P3T_OK : P3T_ERR_CUDA;
}
