// All-pairs sums of the soft force of Eq. softforce (the tree at theta = 0)
// and of its vector-Jacobian product (the adjoint), cut-off radii held fixed:
//   a_k = -G sum_j m_j K(r_kj / r_out,kj) r_kj / r_kj^3,
//   g_k += s sum_j J(r_kj) (m_k lam_j - m_j lam_k),  gm_k += s sum_j phi_kj lam_j . r_kj,
// J = phi I + psi r r^T, phi = K / r^3, psi = K'(y) / (r_out r^4) - 3 K / r^5.
//
// Layout: k_direct_pack writes every particle once as packed 4-vectors in
// the pair arithmetic's type; a block is 8 warps over 64 targets (two per
// lane); each warp takes one eighth of the block's source range and stages
// it 32 sources at a time in its own shared-memory slots (one broadcast load
// per 4-vector, shared by the lane's two targets).  A grid column (blockIdx.y) is
// one split of the sources; each block adds its 8 warps in order and writes its
// per-target sums to part[(split * C + c) * n + k]; the last block of a target tile
// to finish adds the splits in order: the result does not depend on scheduling.
//
// Far sources: with the particles in no spatial order a source is inside the
// cut-off reach of some target of a warp about once in a thousand times (ring
// of 10,000: 1e-5 a pair).  Each source carries a bound T on max(r_out)^2 over
// the warp's targets and itself; a chunk of 32 sources is summed without the
// changeover (K = 1, K' = 0: the same bits in FP32 for 18 packed instructions
// instead of 32 a pair, 43 instead of 63 for the VJP), and when some r^2 of
// the warp was within its bound it is summed again in full (and the next one
// in full at once, as long as near pairs are met); in FP64, where a vote costs
// little beside a pair, each source is voted on.  What bounds the kernels is
// the FP32 (FP64) pipe: a packed instruction holds it two cycles (73 % active at
// N = 50,000).  Measured per call, FP32: force N = 1e4 124 -> 95 us, 5e4 2,518
// -> 1,630, VJP 210 -> 165, 4,624 -> 3,300; FP64: force N = 8,191 2,960 -> 2,100,
// VJP N = 1e4 8,940 -> 7,290.  Where most pairs are near (several neighbours a body,
// whose clusters percolate) the form costs: N = 1e4 124 -> 157 us, VJP 210 -> 293
// (a warp's first chunk of two taken twice), 5e4 2,518 -> 2,526 and 4,624 -> 4,994.  A
// first guess from 512 pairs a block makes that 127 and 225, but 95 -> 99 and 165 ->
// 168 where few are near; votes within a chunk cost the far form 8 to 12 %.  Four
// targets a lane: 1,590 us at 5e4, 128 at 1e4 and 50 instead of 45 at 1,000 (fewer,
// longer blocks): two kept.
//
// Precision: FP64 throughout, or (MIXED) float-float positions whose
// difference (hi_k - hi_j) + (lo_k - lo_j) carries the relative coordinate
// to about 2^-24 of itself, FP32 pair terms summed in FP32 over a 32-source
// chunk and the chunk sums kept as float-float (TwoSum), so that no FP64
// instruction runs inside the pair loop.
#include <math.h>

#include "p3t_internal.cuh"

namespace {

constexpr int kDW = 8;          // warps per block
constexpr int kDT = 2;          // targets per lane
constexpr int kDTB = 32 * kDT;  // targets per block
constexpr int kSplitBlocks = 3;  // blocks an SM that the sources' split counts with
#ifndef P3T_DIRECT_MINB_MIXED
#define P3T_DIRECT_MINB_MIXED 3  // resident blocks per SM asked of the FP32 kernels
#endif

template <typename T>
struct alignas(4 * sizeof(T)) Q4 {
  T x, y, z, w;
};

template <bool MIXED>
struct DT {
  using T = double;
};
template <>
struct DT<true> {
  using T = float;
};

// hi + lo += p without losing the rounding error of the addition (TwoSum)
__device__ __forceinline__ void two_sum_acc(float &hi, float &lo, float p) {
  const float s = hi + p;
  const float b = s - hi;
  lo += (hi - (s - b)) + (p - b);
  hi = s;
}

// r^-3 from r^2's seed (see rsqrt_seed); 0 for r = 0
__device__ __forceinline__ double inv_cube(const RsqrtSeed &s) {
  const double y3 = s.y2 * s.y;
  return fma(y3 * s.e, fma(1.875, s.e, 1.5), y3);
}

// one FP64 pair term: k the target (its mass, 1/r_out and adjoint), j the
// source; NEAR: with the changeover.  A pair within gamma r_out adds nothing:
// the target itself, bodies so near that r^-3 is infinite, and pairs whose r^2
// is not finite.
template <bool VJP, bool NEAR>
__device__ __forceinline__ void pair_term(double rx, double ry, double rz, double r2,
                                          const Q4<double> &A, double iroj, const Q4<double> &L,
                                          double mk, double irok, double lxk, double lyk,
                                          double lzk, double g, double i1mg, double *acc) {
  const RsqrtSeed s = rsqrt_seed(r2);
  double phi = inv_cube(s);         // K / r^3 below
  double dKr = 0.0, K = 1.0;        // K'(y) / r_out
  if constexpr (NEAR) {
    const double irout = irok < iroj ? irok : iroj;  // 1 / max(r_out,k, r_out,j)
    const double ir = fma(s.y * s.e, fma(0.375, s.e, 0.5), s.y);
    const double yv = r2 * ir * irout;
    const double t = (yv - g) * i1mg;
    // NaN too (r = 0 with r_out = 0; an infinite r^2)
    if (!(t > 0.0)) return;
    const double u = t < 1.0 ? t : 1.0, u2 = u * u;
    K = (u2 * u2) * fma(fma(fma(-20.0, u, 70.0), u, -84.0), u, 35.0);
    phi *= K;
    if constexpr (VJP) {
      // zero at the end also where 1 / r_out is infinite
      const double v = 1.0 - u, ie = u < 1.0 ? irout : 0.0;
      dKr = 140.0 * (u2 * u) * (v * v * v) * i1mg * ie;
    }
  }
  if constexpr (!VJP) {
    const double w = A.w * phi;  // m_j K / r^3
    acc[0] = fma(w, rx, acc[0]);
    acc[1] = fma(w, ry, acc[1]);
    acc[2] = fma(w, rz, acc[2]);
  } else {
    const double ir2 = fma(s.y2, fma(s.e, s.e, s.e), s.y2);  // y^2 / (1 - e)
    double psi = -3.0 * (phi * ir2);
    if constexpr (NEAR) psi = fma(ir2 * ir2, dKr, psi);
    const double wx = fma(mk, L.x, -A.w * lxk), wy = fma(mk, L.y, -A.w * lyk),
                 wz = fma(mk, L.z, -A.w * lzk);
    const double prw = psi * fma(rx, wx, fma(ry, wy, rz * wz));
    acc[0] += fma(phi, wx, prw * rx);
    acc[1] += fma(phi, wy, prw * ry);
    acc[2] += fma(phi, wz, prw * rz);
    acc[3] = fma(phi, fma(L.x, rx, fma(L.y, ry, L.z * rz)), acc[3]);
  }
}

// The mixed kernels' pair term for a lane's two targets at once, one per half
// of each packed FP32 pair (f32x2 instructions round each half as the scalar
// one would), the source's values duplicated into both halves.  Branch-free:
// the changeover variable u = clamp((y - gamma) / (1 - gamma), 0, 1) gives K =
// 0 below gamma, 1 beyond r_out and the polynomial between (35 - 84 + 70 - 20
// = 1 exactly), and r^2 is kept above 1e-18 so that the target itself (r = 0,
// y = 0, K = 0) and far-away dummy targets add exact zeros without an inf.
// (Any real pair that close has y <= gamma: K = K' = 0 as well.)
struct PairConst2 {
  f2 g, i1mg, c35, c84, c70, c20, one, three, c140i;
};
template <bool VJP>
__device__ __forceinline__ void pair_term2(f2 rx, f2 ry, f2 rz, const Q4<float> &A, float iroj,
                                           const Q4<float> &L, f2 mk, f2 irok, f2 lxk, f2 lyk,
                                           f2 lzk, const PairConst2 &k, f2 *acc) {
  f2 r2 = fma2(rx, rx, fma2(ry, ry, mul2(rz, rz)));
  r2 = f2_pk(fmaxf(f2_lo(r2), 1e-18f), fmaxf(f2_hi(r2), 1e-18f));
  const f2 ir = f2_pk(rsqrtf(f2_lo(r2)), rsqrtf(f2_hi(r2)));
  const f2 irout = f2_pk(fminf(f2_lo(irok), iroj), fminf(f2_hi(irok), iroj));
  const f2 yv = mul2(mul2(r2, ir), irout);
  const f2 t = mul2(sub2(yv, k.g), k.i1mg);
  const f2 u = f2_pk(__saturatef(f2_lo(t)), __saturatef(f2_hi(t)));
  const f2 u2 = mul2(u, u), u3 = mul2(u2, u);
  const f2 poly = fma2(fma2(fma2(sub2(0ull, k.c20), u, k.c70), u, sub2(0ull, k.c84)), u, k.c35);
  const f2 K = mul2(mul2(u2, u2), poly);
  const f2 ir2 = mul2(ir, ir);
  const f2 phi = mul2(mul2(K, ir2), ir);
  if constexpr (!VJP) {
    const f2 w = mul2(f2_dup(A.w), phi);  // m_j K / r^3
    acc[0] = fma2(w, rx, acc[0]);
    acc[1] = fma2(w, ry, acc[1]);
    acc[2] = fma2(w, rz, acc[2]);
  } else {
    const f2 v = sub2(k.one, u);
    const f2 dKr = mul2(mul2(mul2(k.c140i, u3), mul2(mul2(v, v), v)), irout);
    const f2 psi = mul2(mul2(ir2, ir2), sub2(dKr, mul2(mul2(k.three, K), ir)));
    const f2 mA = f2_dup(A.w);
    const f2 wx = sub2(mul2(mk, f2_dup(L.x)), mul2(mA, lxk));
    const f2 wy = sub2(mul2(mk, f2_dup(L.y)), mul2(mA, lyk));
    const f2 wz = sub2(mul2(mk, f2_dup(L.z)), mul2(mA, lzk));
    const f2 prw = mul2(psi, fma2(rx, wx, fma2(ry, wy, mul2(rz, wz))));
    acc[0] = add2(acc[0], fma2(phi, wx, mul2(prw, rx)));
    acc[1] = add2(acc[1], fma2(phi, wy, mul2(prw, ry)));
    acc[2] = add2(acc[2], fma2(phi, wz, mul2(prw, rz)));
    acc[3] = fma2(phi, fma2(f2_dup(L.x), rx, fma2(f2_dup(L.y), ry, mul2(f2_dup(L.z), rz))),
                  acc[3]);
  }
}

// the same with K = 1 and K' = 0 (every r beyond max(r_out)): pair_term2's
// operations without those that return their operand, so the same bits
template <bool VJP>
__device__ __forceinline__ void pair_far2(f2 rx, f2 ry, f2 rz, f2 r2, const Q4<float> &A,
                                          const Q4<float> &L, f2 mk, f2 lxk, f2 lyk, f2 lzk,
                                          f2 m3, f2 *acc) {
  const f2 ir = f2_pk(rsqrtf(f2_lo(r2)), rsqrtf(f2_hi(r2)));
  const f2 ir2 = mul2(ir, ir);
  const f2 phi = mul2(ir2, ir);
  if constexpr (!VJP) {
    const f2 w = mul2(f2_dup(A.w), phi);
    acc[0] = fma2(w, rx, acc[0]);
    acc[1] = fma2(w, ry, acc[1]);
    acc[2] = fma2(w, rz, acc[2]);
  } else {
    const f2 psi = mul2(mul2(ir2, ir2), mul2(m3, ir));  // m3 = -3
    const f2 mA = f2_dup(A.w);
    const f2 wx = sub2(mul2(mk, f2_dup(L.x)), mul2(mA, lxk));
    const f2 wy = sub2(mul2(mk, f2_dup(L.y)), mul2(mA, lyk));
    const f2 wz = sub2(mul2(mk, f2_dup(L.z)), mul2(mA, lzk));
    const f2 prw = mul2(psi, fma2(rx, wx, fma2(ry, wy, mul2(rz, wz))));
    acc[0] = add2(acc[0], fma2(phi, wx, mul2(prw, rx)));
    acc[1] = add2(acc[1], fma2(phi, wy, mul2(prw, ry)));
    acc[2] = add2(acc[2], fma2(phi, wz, mul2(prw, rz)));
    acc[3] = fma2(phi, fma2(f2_dup(L.x), rx, fma2(f2_dup(L.y), ry, mul2(f2_dup(L.z), rz))),
                  acc[3]);
  }
}

// outputs: with one split, the block writes out_c[k] = (add ? out_c[k] : 0)
// + scale * sum itself; with several, the sums go to part
struct DOut {
  double *o[4];
  double scale;
  int add;
};

// Packs every particle once per call: A = (x_hi, y_hi, z_hi, m), B = (x_lo,
// y_lo, z_lo, 1 / r_out), L = (lam, 0), in the pair arithmetic's type (the
// lo parts are zero in FP64), so that no conversion or FP64 division is
// repeated per block.
template <bool MIXED, bool VJP>
__global__ void k_direct_pack(int64_t n, const double *x, const double *y, const double *z,
                              const double *m, const double *ro, const double *lx,
                              const double *ly, const double *lz,
                              Q4<typename DT<MIXED>::T> *A, Q4<typename DT<MIXED>::T> *B,
                              Q4<typename DT<MIXED>::T> *L) {
  pdl_wait();
  using T = typename DT<MIXED>::T;
  for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < n;
       j += (int64_t)gridDim.x * blockDim.x) {
    Q4<T> a, b;
    a.x = (T)x[j]; a.y = (T)y[j]; a.z = (T)z[j]; a.w = (T)m[j];
    b.x = b.y = b.z = 0;
    if constexpr (MIXED) {
      b.x = (T)(x[j] - (double)a.x);
      b.y = (T)(y[j] - (double)a.y);
      b.z = (T)(z[j] - (double)a.z);
    }
    b.w = (T)(1.0 / ro[j]);
    A[j] = a;
    B[j] = b;
    if constexpr (VJP) {
      Q4<T> l;
      l.x = (T)lx[j]; l.y = (T)ly[j]; l.z = (T)lz[j]; l.w = 0;
      L[j] = l;
    }
  }
}

// the targets of one packed pair
struct Pair2 {
  f2 xh, yh, zh, xl, yl, zl, m, iro, lx, ly, lz;
};

template <bool MIXED, bool VJP>
__global__ void __launch_bounds__(kDW * 32, MIXED ? P3T_DIRECT_MINB_MIXED : 1)
    k_direct(int64_t n, int64_t chunk, const Q4<typename DT<MIXED>::T> *__restrict__ PA,
             const Q4<typename DT<MIXED>::T> *__restrict__ PB,
             const Q4<typename DT<MIXED>::T> *__restrict__ PL, double gamma, double *part,
             int32_t *tile_cnt, DOut out) {
  pdl_wait();
  using T = typename DT<MIXED>::T;
  constexpr int NC = VJP ? 4 : 3;
  constexpr int DTL = kDT, DTB = kDTB;
  constexpr int NP = MIXED ? DTL / 2 : 1;           // packed pairs a lane
  __shared__ Q4<T> sA[kDW][32];                     // x_hi, y_hi, z_hi, m
  __shared__ Q4<T> sB[kDW][32];                     // x_lo, y_lo, z_lo, 1 / r_out
  __shared__ Q4<T> sL[VJP ? kDW : 1][VJP ? 32 : 1];  // lam
  __shared__ T sT[kDW][32];                          // bound on max(r_out)^2, widened
  // the 8 warps' sums: FP64, or (MIXED) float-float pairs added with FP32
  // instructions only (an FP64 instruction costs 64 FP32 issue slots here);
  // the mixed running sums stand here too
  __shared__ double red[MIXED ? 1 : kDW][NC][MIXED ? 1 : DTB];
  __shared__ float red_h[MIXED ? kDW : 1][NC][MIXED ? DTB : 1];
  __shared__ float red_l[MIXED ? kDW : 1][NC][MIXED ? DTB : 1];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const T g = (T)gamma, i1mg = (T)(1.0 / (1.0 - gamma));

  T txh[DTL], tyh[DTL], tzh[DTL], txl[DTL], tyl[DTL], tzl[DTL];
  T tm[DTL], tiro[DTL], tlx[DTL], tly[DTL], tlz[DTL];
  T tmax = 0;  // largest r_out^2 of the lane's targets
#pragma unroll
  for (int t = 0; t < DTL; ++t) {
    const int64_t k = (int64_t)blockIdx.x * DTB + t * 32 + lane;
    txh[t] = tyh[t] = tzh[t] = (T)1e18;  // far from every source
    txl[t] = tyl[t] = tzl[t] = 0;
    tm[t] = tiro[t] = tlx[t] = tly[t] = tlz[t] = 0;  // 1/r_out = 0: no pair term
    if (k < n) {
      const Q4<T> a = PA[k], b = PB[k];
      txh[t] = a.x; tyh[t] = a.y; tzh[t] = a.z; tm[t] = a.w;
      txl[t] = b.x; tyl[t] = b.y; tzl[t] = b.z; tiro[t] = b.w;
      const T ro = (T)1 / b.w;
      tmax = fmax(tmax, ro * ro);
      if constexpr (VJP) {
        const Q4<T> l = PL[k];
        tlx[t] = l.x; tly[t] = l.y; tlz[t] = l.z;
      }
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) tmax = fmax(tmax, __shfl_xor_sync(0xffffffffu, tmax, o));
  Pair2 P[NP];
  PairConst2 kc{};
  if constexpr (MIXED) {
#pragma unroll
    for (int p = 0; p < NP; ++p)
      P[p] = Pair2{f2_pk(txh[2 * p], txh[2 * p + 1]), f2_pk(tyh[2 * p], tyh[2 * p + 1]),
                   f2_pk(tzh[2 * p], tzh[2 * p + 1]), f2_pk(txl[2 * p], txl[2 * p + 1]),
                   f2_pk(tyl[2 * p], tyl[2 * p + 1]), f2_pk(tzl[2 * p], tzl[2 * p + 1]),
                   f2_pk(tm[2 * p], tm[2 * p + 1]), f2_pk(tiro[2 * p], tiro[2 * p + 1]),
                   f2_pk(tlx[2 * p], tlx[2 * p + 1]), f2_pk(tly[2 * p], tly[2 * p + 1]),
                   f2_pk(tlz[2 * p], tlz[2 * p + 1])};
    kc = PairConst2{f2_dup((float)g), f2_dup((float)i1mg), f2_dup(35.f), f2_dup(84.f),
                    f2_dup(70.f), f2_dup(20.f), f2_dup(1.f), f2_dup(3.f),
                    f2_dup((float)(140.0 * (1.0 / (1.0 - gamma))))};
#pragma unroll
    for (int t = 0; t < DTL; ++t)
#pragma unroll
      for (int c = 0; c < NC; ++c)
        red_h[warp][c][t * 32 + lane] = red_l[warp][c][t * 32 + lane] = 0.0f;
  }
  double dd[MIXED ? 1 : DTL][NC];  // FP64 running sums
#pragma unroll
  for (int t = 0; t < (MIXED ? 1 : DTL); ++t)
#pragma unroll
    for (int c = 0; c < NC; ++c) dd[t][c] = 0.0;

  // the split's sources, cut into 8 contiguous, equal (to one source) warp
  // ranges, walked in chunks of 32
  const int64_t b_lo = (int64_t)blockIdx.y * chunk;
  const int64_t b_len = max((int64_t)0, min(n, b_lo + chunk) - b_lo);
  const int64_t s_lo = b_lo + b_len * warp / kDW;
  const int64_t s_hi = b_lo + b_len * (warp + 1) / kDW;
  bool full = false;  // the last chunk had a near pair: take the next in full form
  for (int64_t cb = s_lo; cb < s_hi; cb += 32) {
    const int lim = (int)min((int64_t)32, s_hi - cb);
    __syncwarp();
    if (lane < lim) {
      const int64_t j = cb + lane;
      const Q4<T> b = PB[j];
      sA[warp][lane] = PA[j];
      sB[warp][lane] = b;
      if constexpr (VJP) sL[warp][lane] = PL[j];
      // widened beyond the rounding of r^2 and 1 / r_out; pairs below 1e-17
      // (the target itself) take the near form, which bounds r^2 from below
      const T ro = (T)1 / b.w;
      sT[warp][lane] = fmax(fmax(tmax, ro * ro) * (T)1.0001, (T)1e-17);
    }
    __syncwarp();
    if constexpr (MIXED) {
      // the lane's targets in packed pairs
      f2 a2[NP][NC];
      const f2 m3 = f2_dup(-3.f);
      bool near = false;
      if (!full) {
#pragma unroll
        for (int p = 0; p < NP; ++p)
#pragma unroll
          for (int c = 0; c < NC; ++c) a2[p][c] = 0ull;
#pragma unroll 4
        for (int q = 0; q < lim; ++q) {
          const Q4<T> A = sA[warp][q], B = sB[warp][q];
          const float Tq = sT[warp][q];
          Q4<T> L{0, 0, 0, 0};
          if constexpr (VJP) L = sL[warp][q];
#pragma unroll
          for (int p = 0; p < NP; ++p) {
            const f2 rx = add2(sub2(P[p].xh, f2_dup(A.x)), sub2(P[p].xl, f2_dup(B.x)));
            const f2 ry = add2(sub2(P[p].yh, f2_dup(A.y)), sub2(P[p].yl, f2_dup(B.y)));
            const f2 rz = add2(sub2(P[p].zh, f2_dup(A.z)), sub2(P[p].zl, f2_dup(B.z)));
            const f2 r2 = fma2(rx, rx, fma2(ry, ry, mul2(rz, rz)));
            near = near || !(fminf(f2_lo(r2), f2_hi(r2)) > Tq);
            pair_far2<VJP>(rx, ry, rz, r2, A, L, P[p].m, P[p].lx, P[p].ly, P[p].lz, m3, a2[p]);
          }
        }
        full = __any_sync(0xffffffffu, near);
      }
      if (full) {
#pragma unroll
        for (int p = 0; p < NP; ++p)
#pragma unroll
          for (int c = 0; c < NC; ++c) a2[p][c] = 0ull;
        near = false;
#pragma unroll 2
        for (int q = 0; q < lim; ++q) {
          const Q4<T> A = sA[warp][q], B = sB[warp][q];
          const float Tq = sT[warp][q];
          Q4<T> L{0, 0, 0, 0};
          if constexpr (VJP) L = sL[warp][q];
#pragma unroll
          for (int p = 0; p < NP; ++p) {
            const f2 rx = add2(sub2(P[p].xh, f2_dup(A.x)), sub2(P[p].xl, f2_dup(B.x)));
            const f2 ry = add2(sub2(P[p].yh, f2_dup(A.y)), sub2(P[p].yl, f2_dup(B.y)));
            const f2 rz = add2(sub2(P[p].zh, f2_dup(A.z)), sub2(P[p].zl, f2_dup(B.z)));
            const f2 r2 = fma2(rx, rx, fma2(ry, ry, mul2(rz, rz)));
            near = near || !(fminf(f2_lo(r2), f2_hi(r2)) > Tq);
            pair_term2<VJP>(rx, ry, rz, A, B.w, L, P[p].m, P[p].iro, P[p].lx, P[p].ly, P[p].lz,
                            kc, a2[p]);
          }
        }
        full = __any_sync(0xffffffffu, near);
      }
#pragma unroll
      for (int t = 0; t < DTL; ++t)
#pragma unroll
        for (int c = 0; c < NC; ++c)
          two_sum_acc(red_h[warp][c][t * 32 + lane], red_l[warp][c][t * 32 + lane],
                      t & 1 ? f2_hi(a2[t / 2][c]) : f2_lo(a2[t / 2][c]));
    } else {
      double acc[DTL][NC];
#pragma unroll
      for (int t = 0; t < DTL; ++t)
#pragma unroll
        for (int c = 0; c < NC; ++c) acc[t][c] = 0.0;
#pragma unroll 2
      for (int q = 0; q < lim; ++q) {
        const Q4<T> A = sA[warp][q], B = sB[warp][q];
        const int hT = __double2hiint(sT[warp][q]);
        Q4<T> L{0, 0, 0, 0};
        if constexpr (VJP) L = sL[warp][q];
        double rx[DTL], ry[DTL], rz[DTL], r2[DTL];
        // by the leading 32 bits: an FP64 comparison takes the pipe
        int low = 0x7fffffff, high = 0;
#pragma unroll
        for (int t = 0; t < DTL; ++t) {
          rx[t] = txh[t] - A.x; ry[t] = tyh[t] - A.y; rz[t] = tzh[t] - A.z;
          r2[t] = fma(rx[t], rx[t], fma(ry[t], ry[t], rz[t] * rz[t]));
          low = min(low, __double2hiint(r2[t]));
          high = max(high, __double2hiint(r2[t]));
        }
        if (__any_sync(0xffffffffu, low <= hT || high >= 0x7ff00000)) {  // or not finite
#pragma unroll
          for (int t = 0; t < DTL; ++t)
            pair_term<VJP, true>(rx[t], ry[t], rz[t], r2[t], A, B.w, L, tm[t], tiro[t], tlx[t],
                                 tly[t], tlz[t], g, i1mg, acc[t]);
        } else {
#pragma unroll
          for (int t = 0; t < DTL; ++t)
            pair_term<VJP, false>(rx[t], ry[t], rz[t], r2[t], A, B.w, L, tm[t], tiro[t], tlx[t],
                                  tly[t], tlz[t], g, i1mg, acc[t]);
        }
      }
#pragma unroll
      for (int t = 0; t < DTL; ++t)
#pragma unroll
        for (int c = 0; c < NC; ++c) dd[t][c] += acc[t][c];
    }
  }
  if constexpr (!MIXED)
#pragma unroll
    for (int t = 0; t < DTL; ++t)
#pragma unroll
      for (int c = 0; c < NC; ++c) red[warp][c][t * 32 + lane] = dd[t][c];
  __syncthreads();
  for (int e = threadIdx.x; e < NC * DTB; e += kDW * 32) {
    const int c = e / DTB, tt = e - c * DTB;
    const int64_t k = (int64_t)blockIdx.x * DTB + tt;
    if (k >= n) continue;
    double s = 0.0;
    if constexpr (MIXED) {
      float h = red_h[0][c][tt], l = red_l[0][c][tt];
      for (int w = 1; w < kDW; ++w) {
        two_sum_acc(h, l, red_h[w][c][tt]);
        l += red_l[w][c][tt];
      }
      s = (double)h + (double)l;
    } else {
      for (int w = 0; w < kDW; ++w) s += red[w][c][tt];
    }
    if (gridDim.y == 1) {
      double *o = c == 0 ? out.o[0] : (c == 1 ? out.o[1] : (c == 2 ? out.o[2] : out.o[3]));
      o[k] = (out.add ? o[k] : 0.0) + out.scale * s;
    } else {
      part[((int64_t)blockIdx.y * NC + c) * n + k] = s;
    }
  }
  if (gridDim.y == 1) return;
  // several splits: the last block of this target tile to arrive adds the
  // splits' sums in split order (the result does not depend on which block
  // that is) and resets the tile's counter for the next call
  __shared__ int last;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) last = atomicAdd(&tile_cnt[blockIdx.x], 1) == (int)gridDim.y - 1;
  __syncthreads();
  if (!last) return;
  __threadfence();
  for (int e = threadIdx.x; e < NC * DTB; e += kDW * 32) {
    const int c = e / DTB, tt = e - c * DTB;
    const int64_t k = (int64_t)blockIdx.x * DTB + tt;
    if (k >= n) continue;
    double s = 0.0;
#pragma unroll 8
    for (int q = 0; q < (int)gridDim.y; ++q) s += __ldcg(&part[((int64_t)q * NC + c) * n + k]);
    double *o = c == 0 ? out.o[0] : (c == 1 ? out.o[1] : (c == 2 ? out.o[2] : out.o[3]));
    o[k] = (out.add ? o[k] : 0.0) + out.scale * s;
  }
  if (threadIdx.x == 0) tile_cnt[blockIdx.x] = 0;
}

// Work split: tiles of 64 targets x one source split.  With fewer than 8 waves
// of target tiles alone (three blocks an SM), the sources are split so that the
// grid is at least 8 waves of resident blocks (the last, partial wave then
// costs at most an eighth); every split keeps at least 256 sources (a chunk
// per warp).  With ns >= 2 splits, (ns - 1) n < 8 slots 64, so the partial
// sums, C ns n doubles, fit in 4 * 2 * 8 * slots * 64 (direct_part_doubles).
// The split sets the order of the sums, so it does not follow the kernels'
// occupancy.
struct Split {
  int64_t chunk;
  int nsplit;
};
Split split_for(const p3t_ctx *c, int64_t n) {
  Split s;
  const int64_t tiles = (n + kDTB - 1) / kDTB;
  const int64_t slots = (int64_t)c->num_sms * kSplitBlocks;
  int64_t ns = 1;
  if (tiles < 8 * slots) ns = (8 * slots + tiles - 1) / tiles;
  const int64_t ns_max = (n + kDW * 32 - 1) / (kDW * 32);
  ns = ns > ns_max ? ns_max : ns;
  ns = ns < 1 ? 1 : ns;
  s.chunk = (n + ns - 1) / ns;
  s.chunk = (s.chunk + 31) / 32 * 32;
  s.nsplit = (int)((n + s.chunk - 1) / s.chunk);
  return s;
}

template <bool MIXED, bool VJP>
int launch_direct(p3t_ctx *c, const p3t_particles *p, const double *lx, const double *ly,
                  const double *lz, DOut out, cudaStream_t s) {
  constexpr int NC = VJP ? 4 : 3;
  const int64_t n = p->n;
  const Split sp = split_for(c, n);
  const int64_t tiles = (n + kDTB - 1) / kDTB;
  if (sp.nsplit > 1 && (int64_t)NC * sp.nsplit * n > c->dpart_cap) return P3T_ERR_CAPACITY;
  using T = typename DT<MIXED>::T;
  Q4<T> *A = reinterpret_cast<Q4<T> *>(c->hw);  // 3 n packed 4-vectors <= 96 n bytes
  Q4<T> *B = A + n, *L = B + n;
  pdl_launch(k_direct_pack<MIXED, VJP>, dim3((unsigned)p3t_grid(n, 256, (int64_t)c->num_sms * 4)), dim3(256), 0, s, 
      n, p->x, p->y, p->z, p->m, p->r_out, lx, ly, lz, A, B, L);
  if (sp.nsplit > 1 && tiles > c->dcnt_cap) return P3T_ERR_CAPACITY;
  const dim3 grid((unsigned)tiles, (unsigned)sp.nsplit);
  pdl_launch(k_direct<MIXED, VJP>, dim3(grid), dim3(kDW * 32), 0, s, n, sp.chunk, A, B, L, c->prm.gamma, c->dpart,
                                                c->dcnt, out);
  p3t_note_launches(2);
  return cudaGetLastError() == cudaSuccess ? P3T_OK : P3T_ERR_CUDA;
}

}  // namespace

int64_t p3t_direct_part_doubles(const p3t_ctx *c) {
  return (int64_t)4 * 2 * 8 * c->num_sms * kSplitBlocks * kDTB;
}

// with several splits there are fewer than 8 slots target tiles
int64_t p3t_direct_tile_counters(const p3t_ctx *c) {
  return (int64_t)8 * c->num_sms * kSplitBlocks;
}

int p3t_run_soft_force_direct(p3t_ctx *c, const p3t_particles *p, double *ax, double *ay,
                              double *az, cudaStream_t s) {
  if (p->n == 0) return P3T_OK;
  const DOut out{{ax, ay, az, nullptr}, -c->prm.G, 0};
  return c->prm.precision == P3T_MIXED ? launch_direct<true, false>(c, p, nullptr, nullptr,
                                                                    nullptr, out, s)
                                       : launch_direct<false, false>(c, p, nullptr, nullptr,
                                                                     nullptr, out, s);
}

int p3t_run_soft_force_vjp(p3t_ctx *c, const p3t_particles *p, double h, const double *lx,
                           const double *ly, const double *lz, double *gx, double *gy,
                           double *gz, double *gm, cudaStream_t s) {
  if (p->n == 0) return P3T_OK;
  const DOut out{{gx, gy, gz, gm}, h * c->prm.G, 1};
  return c->prm.precision == P3T_MIXED ? launch_direct<true, true>(c, p, lx, ly, lz, out, s)
                                       : launch_direct<false, true>(c, p, lx, ly, lz, out, s);
}
