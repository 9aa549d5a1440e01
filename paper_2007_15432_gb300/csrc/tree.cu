// Soft step: cut-off radii, Morton keys and sort, octree
// with monopole + quadrupole moments.  Compiled with -fmad=false: the keys
// and the integer grid geometry must be bit-identical on every IEEE machine.
#include <math.h>

#include <algorithm>

#include "p3t_internal.cuh"
#include "cutoff_math.cuh"
#include "exact_conv.cuh"

namespace {

constexpr int kBlock = 256;

// order-preserving map of doubles to unsigned 64-bit integers
__device__ __forceinline__ unsigned long long ord_bits(double v) {
  unsigned long long b = (unsigned long long)__double_as_longlong(v);
  return (b >> 63) ? ~b : (b | 0x8000000000000000ull);
}
__device__ __forceinline__ double ord_double(unsigned long long b) {
  b = (b >> 63) ? (b & 0x7fffffffffffffffull) : ~b;
  return __longlong_as_double((long long)b);
}

// =========================================================================
// Cut-off radii (Eq. routi2, Eq. rsearch).  Random velocity
// u = v - sqrt(G M_* / |x|) phi_hat (phi_hat: cylindrical azimuth),
// v_ran = rms |u| over radial bins uniform in ln R_cyl.
// =========================================================================
// per segment d: bits[4d] min R, bits[4d + 1] max R, bits[4d + 2], [4d + 3]
// the largest r_out and r_search (shared scheme)
// a block's slice of its segment: blocks [d * slices, (d + 1) * slices) take
// segment d in contiguous slices
__device__ __forceinline__ void seg_slice(const SegView &sv, int slices, int &d, int64_t &a,
                                          int64_t &b) {
  d = (int)(blockIdx.x / slices);
  const int sl = (int)(blockIdx.x % slices);
  const int64_t s0 = seg_lo(sv, d), len = seg_hi(sv, d) - s0;
  a = s0 + len * sl / slices;
  b = s0 + len * (sl + 1) / slices;
}

// The range of R of each segment, as that of R^2 (the correctly rounded root
// is monotone), a block's slice at a time into part; the last block of a
// segment to finish (done, left at zero) reduces the slices and takes the
// roots, and with one segment their logarithms (bits[4], bits[5]; the FP32
// estimate's scale in bits[6]), which every thread of k_cut_u2 formed for itself
// before (FP64 logarithms, more work than the rest of that kernel).  Also
// stores the sort's n.
__global__ void k_cut_range(SegView sv, int slices, const double *x, const double *y,
                            unsigned long long *part, uint32_t *done, unsigned long long *bits,
                            int nb, int64_t *d_n) {
  pdl_wait();
  __shared__ unsigned long long red[2][kBlock / 32];
  __shared__ bool s_last;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
  if (blockIdx.x == 0 && threadIdx.x == 0) *d_n = sv.n;
  int d;
  int64_t a, b;
  seg_slice(sv, slices, d, a, b);
  unsigned long long lo = ~0ull, hi = 0ull;
  for (int64_t i = a + threadIdx.x; i < b; i += blockDim.x) {
    const unsigned long long v = ord_bits(x[i] * x[i] + y[i] * y[i]);
    lo = v < lo ? v : lo;
    hi = v > hi ? v : hi;
  }
  auto reduce = [&]() {
    for (int o = 16; o > 0; o >>= 1) {
      const unsigned long long u = __shfl_xor_sync(0xffffffffu, lo, o);
      const unsigned long long c = __shfl_xor_sync(0xffffffffu, hi, o);
      lo = u < lo ? u : lo;
      hi = c > hi ? c : hi;
    }
  };
  reduce();
  if (lane == 0) { red[0][w] = lo; red[1][w] = hi; }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int q = 1; q < nw; ++q) {
      lo = red[0][q] < lo ? red[0][q] : lo;
      hi = red[1][q] > hi ? red[1][q] : hi;
    }
    part[2 * (int64_t)blockIdx.x] = lo;
    part[2 * (int64_t)blockIdx.x + 1] = hi;
    __threadfence();
    s_last = atomicAdd(&done[d], 1u) == (unsigned)slices - 1;
    if (s_last) done[d] = 0;
  }
  __syncthreads();
  if (!s_last || threadIdx.x >= 32) return;
  __threadfence();
  {
    lo = ~0ull;
    hi = 0ull;
    for (int q = lane; q < slices; q += 32) {
      const unsigned long long *v = part + 2 * ((int64_t)d * slices + q);
      const unsigned long long u = __ldcg(&v[0]), c = __ldcg(&v[1]);
      lo = u < lo ? u : lo;
      hi = c > hi ? c : hi;
    }
    reduce();
    if (lane < 2) {  // lane 0: the smallest, lane 1: the largest
      const double R = sqrt(ord_double(lane == 0 ? lo : hi));
      bits[4 * d + lane] = ord_bits(R);
      bits[4 * d + 2 + lane] = 0ull;
      if (sv.nseg == 1) {
        const double l = log(R);
        bits[4 + lane] = (unsigned long long)__double_as_longlong(l);
        const double lmax = __shfl_sync(0x3u, l, 1);
        if (lane == 0) *reinterpret_cast<float2 *>(&bits[6]) = cut_scale(R, l, lmax, nb);
      }
    }
  }
}

// radial bins of each segment (several segments): their number (as for a
// single system), first global bin and log R range
__global__ void k_cut_segbins(SegView sv, int vran_bins, const unsigned long long *bits,
                              int32_t *seg_nb, int32_t *seg_base, double *seg_l) {
  pdl_wait();
  __shared__ int wsum[32];
  __shared__ int carry;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  if (threadIdx.x == 0) carry = 0;
  __syncthreads();
  for (int base = 0; base < sv.nseg; base += blockDim.x) {
    const int d = base + threadIdx.x;
    int nb = 0;
    if (d < sv.nseg) {
      nb = vran_bins;
      if (nb <= 0) {
        const int64_t t = (seg_hi(sv, d) - seg_lo(sv, d)) / 1000;
        nb = (int)(t < 1 ? 1 : (t > 1024 ? 1024 : t));
      }
      seg_nb[d] = nb;
      seg_l[2 * d] = log(ord_double(bits[4 * d]));
      seg_l[2 * d + 1] = log(ord_double(bits[4 * d + 1]));
    }
    int x = nb;
    for (int o = 1; o < 32; o <<= 1) {
      const int t = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += t;
    }
    if (lane == 31) wsum[warp] = x;
    __syncthreads();
    if (warp == 0) {
      const int w0 = lane < nw ? wsum[lane] : 0;
      int y = w0;
      for (int o = 1; o < 32; o <<= 1) {
        const int t = __shfl_up_sync(0xffffffffu, y, o);
        if (lane >= o) y += t;
      }
      if (lane < nw) wsum[lane] = y - w0;
    }
    __syncthreads();
    const int ex = carry + wsum[warp] + (x - nb);
    if (d < sv.nseg) seg_base[d] = ex;
    __syncthreads();
    if (threadIdx.x == blockDim.x - 1) carry = ex + nb;
    __syncthreads();
  }
}

// What bounds the cut-offs from some 1e5 particles on is the FP64 pipe (19 cycles
// of an SM a warp instruction): 23 FP64 instructions a particle in k_cut_u2 and
// some 40 in k_cut_final, the roots from seeds and the bounds' logarithms once.
// Measured, with CUDA's roots and the logarithms a thread, and now, at N = 377,740:
// k_cut_u2 108 -> 27 us, k_cut_final 52 -> 33, k_cut_range 18 -> 14, the whole 213
// -> 104; below, the launches: N = 1,000 43 -> 32 us, 1e5 92 -> 52, 1e6 378 -> 205.
// |u|^2 and the radial bin of every particle (kept for k_cut_final); (bin,
// index) pairs for a stable sort by bin
constexpr int kMaxBins = 4096;
__global__ void k_cut_u2(SegView sv, const double *x, const double *y, const double *z,
                         const double *vx, const double *vy, const double *vz, double smu,
                         const unsigned long long *bits, int nb, const int32_t *seg_nb,
                         const int32_t *seg_base, const double *seg_l, double *u2,
                         uint64_t *key, int32_t *idx, int32_t *bin) {
  pdl_wait();
  const int64_t n = sv.n;
  // one segment: its range here; several: per particle below
  const double Rmin0 = ord_double(bits[0]), Rmax0 = ord_double(bits[1]);
  double lmin0 = 0.0, lmax0 = 0.0;
  float2 sc0 = make_float2(0.f, 0.f);
  if (sv.nseg == 1) {
    sc0 = *reinterpret_cast<const float2 *>(&bits[6]);
    lmin0 = __longlong_as_double((long long)bits[4]);
    lmax0 = __longlong_as_double((long long)bits[5]);
  }
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    const double X = x[i], Y = y[i], Z = z[i];
    const double R2 = X * X + Y * Y;
    // u = v - sqrt(mu / r) phi_hat, phi_hat = (-y, x) / R
    const double t = smu * inv_root4(__fma_rn(Z, Z, R2)) * inv_sqrt(R2);
    const double ux = __fma_rn(t, Y, vx[i]), uy = __fma_rn(-t, X, vy[i]), uz = vz[i];
    u2[i] = __fma_rn(ux, ux, __fma_rn(uy, uy, uz * uz));
    int k;
    if (sv.nseg == 1) {
      k = cut_bin(R2, sc0, Rmin0, Rmax0, lmin0, lmax0, nb);
    } else {
      const int d = seg_of(sv, i);
      const double lmin = seg_l[2 * d], lmax = seg_l[2 * d + 1];
      const double Rmin = ord_double(bits[4 * d]);
      k = seg_base[d] + cut_bin(R2, cut_scale(Rmin, lmin, lmax, seg_nb[d]), Rmin,
                                ord_double(bits[4 * d + 1]), lmin, lmax, seg_nb[d]);
    }
    key[i] = (uint64_t)k;
    idx[i] = (int32_t)i;
    bin[i] = k;
  }
}

// first place of sorted keys that is not below k, by a warp
__device__ __forceinline__ int64_t lower_bound_warp(const uint64_t *keys, int64_t n, uint64_t k) {
  const int lane = threadIdx.x & 31;
  int64_t lo = 0, len = n;
  while (len > 0) {  // shrinks to at most a 32nd
    const int64_t step = (len + 31) >> 5, p = lane * step;
    const unsigned below = __ballot_sync(0xffffffffu, p < len && keys[lo + p] < k);
    if (below == 0) break;
    const int64_t past = (int64_t)(__popc(below) - 1) * step + 1;
    lo += past;
    len = step - 1 < len - past ? step - 1 : len - past;
  }
  return lo;
}

// v_ran of each bin, sqrt(sum |u|^2 / count), the sum by one warp per bin
// over its members in index order (a fixed lane-strided order and a fixed
// shuffle tree: the same sum on every run), the loads of eight members a lane
// at a time before their additions.  The bins' ends by search in the sorted
// bins: counted instead, every block of k_cut_u2 added every bin to the same
// few words.
__global__ void k_cut_binsum(int nb, int64_t n, const uint64_t *sorted_bin,
                             const int32_t *sorted_idx, const double *u2, double *bvr) {
  pdl_wait();
  const int lane = threadIdx.x & 31;
  const int64_t w0 = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t k = w0; k < nb; k += nw) {
    const int64_t b0 = lower_bound_warp(sorted_bin, n, (uint64_t)k);
    const int64_t b1 = lower_bound_warp(sorted_bin, n, (uint64_t)k + 1);
    double sum = 0.0;
    int64_t j = b0 + lane;
    for (; j + 7 * 32 < b1; j += 8 * 32) {
      double v[8];
#pragma unroll
      for (int q = 0; q < 8; ++q) v[q] = u2[sorted_idx[j + 32 * q]];
#pragma unroll
      for (int q = 0; q < 8; ++q) sum += v[q];
    }
    for (; j < b1; j += 32) sum += u2[sorted_idx[j]];
    for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
    if (lane == 0) bvr[k] = sqrt(sum / (double)(b1 - b0));
  }
}

__global__ void k_cut_final(SegView sv, const double *x, const double *y,
                            const double *z, const double *vx, const double *vy,
                            const double *vz, const double *m, p3t_params prm, double imu,
                            double i3ms, unsigned long long *bits, const int32_t *bin,
                            const double *bvr, double *r_out, double *r_search) {
  pdl_wait();
  const int64_t n = sv.n;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    const double r2 = __fma_rn(x[i], x[i], __fma_rn(y[i], y[i], z[i] * z[i]));
    const double ir = inv_sqrt(r2);
    const double v2 = __fma_rn(vx[i], vx[i], __fma_rn(vy[i], vy[i], vz[i] * vz[i]));
    const double alpha = __fma_rn(-v2, imu, 2.0 * ir);  // 1/a, vis-viva
    const double a = alpha > 0.0 ? 1.0 / alpha : r2 * ir;
    double rhill = cbrt_pos(m[i] * i3ms) * a;
    const double vr = bvr[bin[i]];
    // Eq. routi2 (P3T_CUT_HILL_VRAN) or Eq. routi (the other two); Eq. rsearch
    const double ro = prm.cutoff_mode == P3T_CUT_HILL_VRAN
                          ? fmax(prm.rcut0 * rhill, prm.rcut1 * vr * prm.dt_soft)
                          : prm.rcut0 * rhill;
    const double rs = prm.rs0 * ro + prm.rs1 * vr * prm.dt_soft;
    r_out[i] = ro;
    r_search[i] = rs;
    if (prm.cutoff_mode == P3T_CUT_SHARED) {
      // non-negative doubles order like their bit patterns
      const int d = seg_at(sv, i);
      atomicMax(&bits[4 * d + 2], (unsigned long long)__double_as_longlong(ro));
      atomicMax(&bits[4 * d + 3], (unsigned long long)__double_as_longlong(rs));
    }
  }
}

// shared cut-off (Eq. rout1): every particle gets the largest r_out and the
// largest search radius
__global__ void k_cut_shared(SegView sv, const unsigned long long *bits, double *r_out,
                             double *r_search) {
  pdl_wait();
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < sv.n;
       i += (int64_t)gridDim.x * blockDim.x) {
    const int d = seg_at(sv, i);
    r_out[i] = __longlong_as_double((long long)bits[4 * d + 2]);
    r_search[i] = __longlong_as_double((long long)bits[4 * d + 3]);
  }
}

// =========================================================================
// Keys, sort, octree, moments.
// =========================================================================
// min / max of the positions of each segment: warp and block reductions over
// a block's slice of its segment into part; the last block of a segment to
// finish (done, left at zero) reduces the slices to its root cube: corner at
// the per-axis minimum, side = largest extent; box[5 d ..]: corner, side L,
// quantisation scale S
__global__ void k_box(SegView sv, int slices, const double *x, const double *y,
                      const double *z, unsigned long long *part, uint32_t *done, double *box5) {
  pdl_wait();
  __shared__ unsigned long long red[6][kBlock / 32];
  __shared__ bool s_last;
  int d;
  int64_t sa, sb;
  seg_slice(sv, slices, d, sa, sb);
  unsigned long long lo[3] = {~0ull, ~0ull, ~0ull}, hi[3] = {0ull, 0ull, 0ull};
  // four elements a trip, their loads issued before the first is used
  for (int64_t i0 = sa + threadIdx.x; i0 < sb; i0 += 4 * (int64_t)blockDim.x) {
    double v[4][3];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int64_t i = i0 + k * (int64_t)blockDim.x;
      if (i < sb) { v[k][0] = x[i]; v[k][1] = y[i]; v[k][2] = z[i]; }
    }
#pragma unroll
    for (int k = 0; k < 4; ++k)
      if (i0 + k * (int64_t)blockDim.x < sb) {
#pragma unroll
        for (int a = 0; a < 3; ++a) {
          const unsigned long long b = ord_bits(v[k][a]);
          lo[a] = b < lo[a] ? b : lo[a];
          hi[a] = b > hi[a] ? b : hi[a];
        }
      }
  }
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    for (int o = 16; o > 0; o >>= 1) {
      unsigned long long u = __shfl_xor_sync(0xffffffffu, lo[a], o);
      unsigned long long v = __shfl_xor_sync(0xffffffffu, hi[a], o);
      lo[a] = u < lo[a] ? u : lo[a];
      hi[a] = v > hi[a] ? v : hi[a];
    }
    if ((threadIdx.x & 31) == 0) { red[a][threadIdx.x >> 5] = lo[a]; red[3 + a][threadIdx.x >> 5] = hi[a]; }
  }
  __syncthreads();
  if (threadIdx.x < 6) {
    const int a = threadIdx.x;
    unsigned long long r = red[a][0];
    for (int w = 1; w < (int)(blockDim.x >> 5); ++w)
      r = a < 3 ? (red[a][w] < r ? red[a][w] : r) : (red[a][w] > r ? red[a][w] : r);
    part[6 * (int64_t)blockIdx.x + a] = r;
    __threadfence();
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    s_last = atomicAdd(&done[d], 1u) == (unsigned)slices - 1;
    if (s_last) done[d] = 0;
  }
  __syncthreads();
  if (!s_last || threadIdx.x >= 32) return;
  __threadfence();
  const int lane = threadIdx.x;
  {
    unsigned long long mn[3] = {~0ull, ~0ull, ~0ull}, mx[3] = {0ull, 0ull, 0ull};
    for (int q = lane; q < slices; q += 32) {
      const unsigned long long *v = part + 6 * ((int64_t)d * slices + q);
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        const unsigned long long l = __ldcg(&v[a]), h = __ldcg(&v[3 + a]);
        mn[a] = l < mn[a] ? l : mn[a];
        mx[a] = h > mx[a] ? h : mx[a];
      }
    }
#pragma unroll
    for (int a = 0; a < 3; ++a)
      for (int o = 16; o > 0; o >>= 1) {
        const unsigned long long l = __shfl_xor_sync(0xffffffffu, mn[a], o);
        const unsigned long long h = __shfl_xor_sync(0xffffffffu, mx[a], o);
        mn[a] = l < mn[a] ? l : mn[a];
        mx[a] = h > mx[a] ? h : mx[a];
      }
    if (lane == 0) {
      double *box = box5 + 5 * d;
      double lo0[3], hi0[3];
      for (int a = 0; a < 3; ++a) { lo0[a] = ord_double(mn[a]); hi0[a] = ord_double(mx[a]); }
      double L = fmax(hi0[0] - lo0[0], fmax(hi0[1] - lo0[1], hi0[2] - lo0[2]));
      if (!(L > 0.0)) L = 1.0;
      box[0] = lo0[0]; box[1] = lo0[1]; box[2] = lo0[2]; box[3] = L;
      box[4] = (double)P3T_QMAX / L;  // quantisation scale S
    }
  }
}

__device__ __forceinline__ uint64_t spread3(uint64_t v) {
  v &= 0x1fffffull;
  v = (v | (v << 32)) & 0x1f00000000ffffull;
  v = (v | (v << 16)) & 0x1f0000ff0000ffull;
  v = (v | (v << 8)) & 0x100f00f00f00f00full;
  v = (v | (v << 4)) & 0x10c30c30c30c30c3ull;
  v = (v | (v << 2)) & 0x1249249249249249ull;
  return v;
}
__device__ __forceinline__ uint32_t compact3(uint64_t v) {
  v &= 0x1249249249249249ull;
  v = (v ^ (v >> 2)) & 0x10c30c30c30c30c3ull;
  v = (v ^ (v >> 4)) & 0x100f00f00f00f00full;
  v = (v ^ (v >> 8)) & 0x1f0000ff0000ffull;
  v = (v ^ (v >> 16)) & 0x1f00000000ffffull;
  v = (v ^ (v >> 32)) & 0x1fffffull;
  return (uint32_t)v;
}

// Morton key of each particle on its segment's grid.  rekey = 0: slot s holds
// particle s (idx[s] = s), and the particle's record (x, y, z, m, r_out,
// r_search) is packed for the gather (one 48-byte read per particle there in
// place of six scattered 8-byte ones); rekey = 1: slot s holds particle idx[s]
// (the keys of an order already sorted)
__global__ void k_keys(SegView sv, const double *x, const double *y,
                       const double *z, const double *m, const double *ro,
                       const double *rs, const double *box5, uint64_t *keys,
                       int32_t *idx, double *pack, int rekey, int64_t *d_n) {
  pdl_wait();
  const int64_t n = sv.n;
  if (d_n && blockIdx.x == 0 && threadIdx.x == 0) *d_n = n;  // for the count-driven primitives
  for (int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; s < n;
       s += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = rekey ? (int64_t)idx[s] : s;
    const double *box = box5 + 5 * seg_at(sv, i);
    const CellScale cs = cell_scale(box[3]);
    const double X = x[i], Y = y[i], Z = z[i];
    const uint64_t qx = quantise(X, box[0], cs), qy = quantise(Y, box[1], cs),
                   qz = quantise(Z, box[2], cs);
    keys[s] = (spread3(qx) << 2) | (spread3(qy) << 1) | spread3(qz);
    if (!rekey) {
      idx[s] = (int32_t)s;
      double2 *o = reinterpret_cast<double2 *>(pack + 6 * s);
      o[0] = make_double2(X, Y);
      o[1] = make_double2(Z, m[s]);
      o[2] = make_double2(ro[s], rs[s]);
    }
  }
}

// the segment of the particle in each slot, as the key of a stable sort
// that brings each segment's particles together in key order
__global__ void k_segkey(SegView sv, const int32_t *idx, uint64_t *keys) {
  pdl_wait();
  for (int64_t s = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; s < sv.n;
       s += (int64_t)gridDim.x * blockDim.x)
    keys[s] = (uint64_t)seg_of(sv, idx[s]);
}

// common prefix of two keys in levels (0..21)
__device__ __forceinline__ int lcp_levels(uint64_t a, uint64_t b) {
  uint64_t d = a ^ b;
  if (d == 0) return P3T_BITS;
  return (__clzll((long long)d) - 1) / 3;
}

// Per sorted particle, a tile of a block's threads at a time:
//  - the sorted copies: the FP64 arrays the FP64 path reads, or the float-float
//    packing the mixed path reads (each path writes only its own);
//  - its common prefix with its predecessor (lp, levels; -1 at a segment's
//    first particle), its leaf level and the number of nodes it starts.  The
//    cell of i at level l holds more than `leaf` particles iff some window of
//    leaf + 1 consecutive sorted particles containing i (within its segment)
//    shares the level-l prefix; the window prefixes w(a) = lcp(a, a + leaf) of
//    the tile and the `leaf` positions before it are formed once in shared
//    memory.  (Each segment's particles are a contiguous sorted run with a
//    tree of its own.)
constexpr int kLevelTile = 256;  // = kBlock
template <bool MIXED>
__global__ void __launch_bounds__(kLevelTile)
k_gather(SegView sv, const int32_t *idx, const uint64_t *keys, const double *pack, double *sx,
         double *sy, double *sz, double *sm, double *sro, double *srs, int32_t *sq, float4 *spA,
         float4 *spB, float *srs32, float *sml, int leaf, int8_t *lp, int8_t *lv,
         int32_t *ncount) {
  pdl_wait();
  __shared__ int8_t w[kLevelTile + 32];  // leaf <= 32
  const int64_t n = sv.n;
  for (int64_t t0 = (int64_t)blockIdx.x * kLevelTile; t0 < n;
       t0 += (int64_t)gridDim.x * kLevelTile) {
    const int64_t s = t0 + threadIdx.x;
    double2 r0, r1, r2;
    uint64_t k = 0;
    if (s < n) {  // the record's loads are in flight during the window prefixes
      const double2 *rec = reinterpret_cast<const double2 *>(pack + 6 * (int64_t)idx[s]);
      r0 = rec[0]; r1 = rec[1]; r2 = rec[2];
      k = keys[s];
    }
    __syncthreads();
    for (int j = threadIdx.x; j < kLevelTile + leaf; j += kLevelTile) {
      const int64_t a = t0 - leaf + j;
      w[j] = (a >= 0 && a + leaf < n) ? (int8_t)lcp_levels(keys[a], keys[a + leaf]) : (int8_t)-1;
    }
    __syncthreads();
    if (s >= n) continue;
    {
      const int d = seg_at(sv, s);
      const int64_t s0 = seg_lo(sv, d), s1 = seg_hi(sv, d);
      const int p = s == s0 ? -1 : lcp_levels(keys[s - 1], k);
      lp[s] = (int8_t)p;
      int D = -1;
      const int64_t a0 = s - leaf > s0 ? s - leaf : s0;
      const int64_t a1 = s < s1 - 1 - leaf ? s : s1 - 1 - leaf;
      for (int64_t a = a0; a <= a1; ++a) D = max(D, (int)w[a - (t0 - leaf)]);
      const int L = min(D + 1, P3T_BITS);
      lv[s] = (int8_t)L;
      ncount[s] = max(0, L - p);
    }
    const double X = r0.x, Y = r0.y, Z = r1.x, M = r1.y, RO = r2.x, RS = r2.y;
    srs[s] = RS;
    sq[3 * s + 0] = (int32_t)compact3(k >> 2);
    sq[3 * s + 1] = (int32_t)compact3(k >> 1);
    sq[3 * s + 2] = (int32_t)compact3(k);
    if constexpr (!MIXED) {
      sx[s] = X; sy[s] = Y; sz[s] = Z; sm[s] = M; sro[s] = RO;
    } else {
      float xh, xl, yh, yl, zh, zl, mh, ml, roh, rol, r2h, r2l;
      split_f32(X, xh, xl);
      split_f32(Y, yh, yl);
      split_f32(Z, zh, zl);
      split_f32(M, mh, ml);
      split_f32(RO, roh, rol);
      split_f32(RS * RS, r2h, r2l);
      spA[s] = make_float4(xh, yh, zh, mh);
      sml[s] = ml;
      spB[s] = make_float4(xl, yl, zl, 1.0f / roh);  // FP32 path only
      srs32[s] = r2h * 1.00001f;  // walk's candidate test: r^2 vs r_search^2, widened
    }
  }
}

// The nodes a particle starts (levels lp + 1 .. lv, deepest last in preorder):
// their first particle and level, and the identity order for the level sort;
// the member counts come from k_node_counts
__global__ void k_nodes_pre(SegView sv, const int8_t *lp, const int8_t *lv,
                            const int64_t *nstart, int64_t *cnt, int64_t node_cap,
                            int32_t *pre_first, int32_t *pre_level, uint64_t *lvl_keys,
                            int32_t *bfs2pre, DevStatus *st) {
  pdl_wait();
  // the node count (cnt[1], from the scan) clamped to the capacity in cnt[3]:
  // the later kernels index with the clamped value
  const int64_t nn = cnt[1];
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    if (nn > node_cap) dev_fail(st, P3T_ERR_CAPACITY, 10, nn);
    cnt[3] = nn < node_cap ? nn : node_cap;
  }
  if (nn > node_cap || st->code != 0) return;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < sv.n;
       i += (int64_t)gridDim.x * blockDim.x) {
    const int l0 = (int)lp[i] + 1, L = (int)lv[i];
    for (int l = l0; l <= L; ++l) {
      const int64_t id = nstart[i] + (l - l0);
      pre_first[id] = (int32_t)i;
      pre_level[id] = l;
      lvl_keys[id] = (uint64_t)l;
      bfs2pre[id] = (int32_t)id;
    }
  }
}

// Members of each node: the node's cell (level l, first particle i) ends at
// the first sorted key at or above kend = (prefix of key i at level l, plus
// one) shifted back, or at the segment's end -- a lower bound found with 8
// independent probes a round: galloping from i (probe steps 1..8, then 8x
// larger each round), then narrowing the last interval ninefold a round.  A
// node's search is its own thread's: the longest chain (the root) is about a
// dozen rounds, not one search per level in a row.
__global__ void k_node_counts(SegView sv, const uint64_t *keys, const int64_t *d_nnode,
                              int64_t node_cap, const int32_t *pre_first,
                              const int32_t *pre_level, int32_t *pre_count, DevStatus *st) {
  pdl_wait();
  if (*d_nnode > node_cap || st->code != 0) return;
  const int64_t nn = *d_nnode;
  for (int64_t b = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; b < nn;
       b += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = pre_first[b];
    const int l = pre_level[b];
    const int64_t s1 = seg_hi(sv, seg_at(sv, i));
    int64_t end = s1;
    if (l > 0) {
      const int sh = 3 * (P3T_BITS - l);
      const uint64_t kend = ((keys[i] >> sh) + 1) << sh;
      // invariant: keys[lo] < kend; the answer lies in (lo, hi]
      int64_t lo = i, hi = s1, step = 1;
      for (;;) {  // gallop
        uint64_t kp[8];
#pragma unroll
        for (int m = 0; m < 8; ++m) {
          const int64_t q = lo + (m + 1) * step;
          kp[m] = q < s1 ? __ldg(&keys[q]) : ~0ull;
        }
        int f = 8;
#pragma unroll
        for (int m = 7; m >= 0; --m)
          if (kp[m] >= kend) f = m;
        if (f < 8) {
          hi = lo + (f + 1) * step < s1 ? lo + (f + 1) * step : s1;
          lo += f * step;
          break;
        }
        lo += 8 * step;
        step *= 8;
      }
      while (hi - lo > 1) {  // narrow (lo, hi]
        const int64_t w = (hi - lo + 8) / 9;
        uint64_t kp[8];
#pragma unroll
        for (int m = 0; m < 8; ++m) {
          const int64_t q = lo + (m + 1) * w;
          kp[m] = q < hi ? __ldg(&keys[q]) : ~0ull;
        }
        int f = 8;
#pragma unroll
        for (int m = 7; m >= 0; --m)
          if (kp[m] >= kend) f = m;
        const int64_t nhi = lo + (f + 1) * w;
        if (nhi < hi) hi = nhi;
        lo += f * w;
      }
      end = hi;
    }
    pre_count[b] = (int32_t)(end - i);
  }
}

// Breadth-first order of the nodes of a small system by one block: the stable
// order by level of the preorder nodes.  A warp takes 32 consecutive nodes at a
// time and counts each level among them by the match of the lanes; a warp a
// level then scans the counts, and the nodes go to their places.  (Larger
// systems take a radix pass: three launches.)
constexpr int kOrderMax = 16384;
__global__ void __launch_bounds__(1024) k_level_order(const int64_t *d_nnode,
                                                      const int32_t *pre_level, int32_t *bfs2pre,
                                                      int32_t *pre2bfs) {
  pdl_wait();
  constexpr int kLevels = P3T_BITS + 1, kGroups = kOrderMax / 32;
  __shared__ uint16_t s_cnt[kLevels][kGroups];  // per level and 32 nodes
  __shared__ int s_tot[kLevels];
  const int nn = (int)*d_nnode, t = threadIdx.x, lane = t & 31, wp = t >> 5;
  const int ng = (nn + 31) >> 5;
  for (int g = wp; g < ng; g += 32) {
    const int id = 32 * g + lane;
    const int l = id < nn ? pre_level[id] : -1;
    const unsigned m = __match_any_sync(0xffffffffu, l);
    if (lane < kLevels) s_cnt[lane][g] = 0;
    __syncwarp();
    if (l >= 0 && lane == __ffs(m) - 1) s_cnt[l][g] = (uint16_t)__popc(m);
  }
  __syncthreads();
  if (wp < kLevels) {
    int run = 0;
    for (int g0 = 0; g0 < ng; g0 += 32) {
      const int c = g0 + lane < ng ? s_cnt[wp][g0 + lane] : 0;
      int v = c;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int u = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += u;
      }
      if (g0 + lane < ng) s_cnt[wp][g0 + lane] = (uint16_t)(run + v - c);
      run += __shfl_sync(0xffffffffu, v, 31);
    }
    if (lane == 0) s_tot[wp] = run;
  }
  __syncthreads();
  int first = 0;  // lane l: the nodes of the levels above l
  for (int l = 0; l < kLevels; ++l)
    if (l < lane) first += s_tot[l];
  for (int g = wp; g < ng; g += 32) {
    const int id = 32 * g + lane;
    const int l = id < nn ? pre_level[id] : -1;
    const unsigned m = __match_any_sync(0xffffffffu, l);
    const int base = __shfl_sync(0xffffffffu, first, l < 0 ? 0 : l);
    if (l < 0) continue;  // the last group's tail: no shuffle follows for it
    const int pos = base + s_cnt[l][g] + __popc(m & ((1u << lane) - 1u));
    bfs2pre[pos] = id;
    pre2bfs[id] = pos;
  }
}

__global__ void k_nodes_bfs(const int64_t *d_nnode, int64_t node_cap,
                            const int32_t *bfs2pre, const int32_t *pre2bfs,
                            const int32_t *pre_first, const int32_t *pre_count,
                            const int32_t *pre_level, const int8_t *lp,
                            const int8_t *lv, const int64_t *nstart,
                            const int32_t *sq, TreeNode *node,
                            int gs, int32_t *flags, int32_t *node_done, DevStatus *st) {
  pdl_wait();
  const int64_t nn = min(*d_nnode, node_cap);
  for (int64_t b = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; b < nn;
       b += (int64_t)gridDim.x * blockDim.x) {
    const int32_t pre = bfs2pre[b];
    const int32_t first = pre_first[pre], count = pre_count[pre], l = pre_level[pre];
    TreeNode nd;
    nd.level = l;
    nd.first = first;
    nd.count = count;
    const int sh = P3T_BITS - l;
    for (int a = 0; a < 3; ++a) nd.c2[a] = (2 * (sq[3 * first + a] >> sh) + 1) << sh;
    const bool internal = l < (int)lv[first];
    if (internal && pre + 1 < nn) {
      nd.child0 = pre2bfs[pre + 1];
      // the children in preorder; each gets its parent link and its flags
      // (bit 0: a leaf; bit 1: a target group, a node holding <= gs particles,
      // or a leaf, whose parent holds more) from here
      const int64_t e = (int64_t)first + count;
      const bool big = count > gs;
      int k = 0;
      int64_t c = pre + 1;
      for (;;) {
        const int32_t cfirst = pre_first[c], ccount = pre_count[c];
        const bool cleaf = l + 1 >= (int)lv[cfirst];
        flags[c] = (cleaf ? 1 : 0) | (big && (ccount <= gs || cleaf) ? 2 : 0);
        if ((int64_t)nd.child0 + k < nn && nd.child0 > b)
          node[nd.child0 + k].parent = (int32_t)b;
        ++k;
        const int64_t cend = (int64_t)cfirst + ccount;
        if (cend >= e) break;
        c = nstart[cend] + (l + 1) - ((int)lp[cend] + 1);
        if (k >= 8 || c <= pre || c >= nn) {  // cannot happen in a consistent tree
          dev_fail(st, P3T_ERR_INVALID, 11, 0);
          break;
        }
      }
      nd.nchild = k;
      node_done[b] = k;
    } else {
      nd.child0 = -1;
      nd.nchild = 0;
      node_done[b] = 0;
    }
    // a root's own flags (a target group when it is small)
    if (l == 0) {
      const bool small = count <= gs || nd.nchild == 0;
      flags[pre] = (internal ? 0 : 1) | (small ? 2 : 0);
    }
    // geometry (qlo, qhi, R) is filled bottom-up by the moments, the parent
    // link by the parent
    TreeNode *o = &node[b];
    o->level = nd.level; o->first = nd.first; o->count = nd.count;
    o->c2[0] = nd.c2[0]; o->c2[1] = nd.c2[1]; o->c2[2] = nd.c2[2];
    o->child0 = nd.child0; o->nchild = nd.nchild;
    if (l == 0) o->parent = -1;
  }
}

// the leaf list and the target-group list in key order from the flag-pair
// scan (leaf positions in bits 0-30, group positions from bit 31), and both
// counts from its total
__global__ void k_lists(const int64_t *d_nnode, int64_t node_cap, const int32_t *flags,
                        const int64_t *pos, const int32_t *pre2bfs, const int64_t *d_total,
                        int32_t *leaf_list, int32_t *group_list, int64_t *d_nleaf,
                        int64_t *d_ngroup) {
  pdl_wait();
  const int64_t nn = min(*d_nnode, node_cap);
  constexpr int64_t kLow = (1ll << 31) - 1;
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    const int64_t t = *d_total;
    *d_nleaf = t & kLow;
    *d_ngroup = t >> 31;
  }
  for (int64_t p = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; p < nn;
       p += (int64_t)gridDim.x * blockDim.x) {
    const int32_t f = flags[p];
    if (!f) continue;
    const int64_t q = pos[p];
    const int32_t b = pre2bfs[p];
    if (f & 1) leaf_list[q & kLow] = b;
    if (f & 2) group_list[q >> 31] = b;
  }
}

// Moments of the FP64 path.  A leaf's members are summed, in their order, about
// a reference point r (its first member): M, D = sum m d, S_ab = sum m d_a d_b
// with d = x - r; then com = r + D / M and the traceless quadrupole about the
// com, Q_ab = 3 C_ab - delta_ab tr C with C_ab = S_ab - M e_a e_b, e = D / M
// (the definition sum m (3 d'_a d'_b - d'^2 delta_ab), d' = x - com,
// expanded).  An internal node sums its children with the parallel-axis shift
// of Q.  What bounds them is the latency of FP64 instructions (64 cycles of a
// sub-partition each, however few lanes are active): a node takes eight lanes,
// and of every sum that the lanes could all form alike each lane forms its own
// part.  Measured (whole FP64 tree build, against a launch a level and a thread
// a leaf): N = 1,000 114 -> 64 us, 1e4 154 -> 107, 1e5 194 -> 152, 1e6 588 -> 458.
__device__ __forceinline__ int64_t max_reach(int64_t a, double v) {  // a NaN is passed over
  const int64_t b = __double_as_longlong(v);
  return b > a && b <= 0x7ff0000000000000ll ? b : a;
}
__device__ __forceinline__ int32_t leaf_moments64_thread(
    int64_t b, TreeNode *node, Mom64 *m64, double *nrs, const double *sx, const double *sy,
    const double *sz, const double *sm, const double *srs, const int32_t *sq, const double *box,
    const SegView &sv) {
  TreeNode *nd = &node[b];
  const int32_t f = nd->first, c = nd->count;
  const double L = box[5 * seg_at(sv, f) + 3];
  const double rx = sx[f], ry = sy[f], rz = sz[f];
  double M = 0.0, D[3] = {0, 0, 0}, S[6] = {0, 0, 0, 0, 0, 0};
  int64_t rsb = 0;
  int32_t lo[3] = {P3T_QMAX, P3T_QMAX, P3T_QMAX}, hi[3] = {-1, -1, -1};
  for (int32_t i = f; i < f + c; ++i) {
    const double m = sm[i], dx = sx[i] - rx, dy = sy[i] - ry, dz = sz[i] - rz;
    const double mx = m * dx, my = m * dy, mz = m * dz;
    M += m; D[0] += mx; D[1] += my; D[2] += mz;
    S[0] = __fma_rn(mx, dx, S[0]); S[1] = __fma_rn(my, dy, S[1]); S[2] = __fma_rn(mz, dz, S[2]);
    S[3] = __fma_rn(mx, dy, S[3]); S[4] = __fma_rn(mx, dz, S[4]); S[5] = __fma_rn(my, dz, S[5]);
    rsb = max_reach(rsb, srs[i]);
#pragma unroll
    for (int a = 0; a < 3; ++a) { lo[a] = min(lo[a], sq[3 * i + a]); hi[a] = max(hi[a], sq[3 * i + a]); }
  }
  Mom64 mm = {};
  const double iM = 1.0 / M;
  const double e[3] = {D[0] * iM, D[1] * iM, D[2] * iM};
  mm.M = M; mm.cx = rx + e[0]; mm.cy = ry + e[1]; mm.cz = rz + e[2];
  const double Cxx = S[0] - M * e[0] * e[0], Cyy = S[1] - M * e[1] * e[1],
               Czz = S[2] - M * e[2] * e[2];
  const double tr = Cxx + Cyy + Czz;
  mm.qxx = 3.0 * Cxx - tr; mm.qyy = 3.0 * Cyy - tr; mm.qzz = 3.0 * Czz - tr;
  mm.qxy = 3.0 * (S[3] - M * e[0] * e[1]);
  mm.qxz = 3.0 * (S[4] - M * e[0] * e[2]);
  mm.qyz = 3.0 * (S[5] - M * e[1] * e[2]);
  for (int a = 0; a < 3; ++a) { nd->qlo[a] = lo[a]; nd->qhi[a] = hi[a]; }
  const double rs = __longlong_as_double(rsb);
  nrs[b] = rs;
  nd->R = reach_cells(rs, L, cell_scale(L));
  m64[b] = mm;
  return nd->parent;
}

// Mixed path: the same moments with no FP64 instruction, written straight to
// the Mom32 record the mixed walk reads (the FP64 record is not formed).
// Positions come as float-float pairs (spA hi, spB lo) and masses as spA.w +
// the lo array; d = x - r, M and D are float-float (the centre of mass then
// carries ~2^-44 of the coordinates, the float-float redo's need), S and the
// quadrupole are FP32 (the walk reads Q in FP32).  The search reach is the
// largest r_search as a bit pattern (non-negative doubles order like their
// bits), and R = ceil(rs / u) + 1 comes from integer operations (reach_cells:
// the value of the FP64 expression the FP64 path evaluates).
__device__ __forceinline__ int64_t max_bits(int64_t a, double v) {
  const int64_t b = __double_as_longlong(v);
  return b > a ? b : a;
}

// What bounds the mixed moments: for few leaves latency (a leaf's serial sums,
// then a chain of a dozen parents, each an atomic, a fence, the children's
// records from L2 and some 400 dependent instructions when one thread does
// it, 4 us a level), for many the leaves' instructions.  A node is therefore
// taken by eight lanes (group mask gm, lane `sub` of the group), a child a
// lane, the children added in the fixed tree by shuffles.  A leaf is taken by
// eight lanes where that fits the resident threads (its members are multiplied
// out one a lane; the sums, serial in the member order, are dealt to the
// lanes from shared memory) and by one thread above (eight lanes for all: 233
// us at N = 1e6).  The same operations in the same order in every form.
// Measured (whole mixed tree build): N = 3,001 96 -> 84 us, 1e5 146 -> 130, 1e6
// 330 -> 326; one thread a leaf throughout 91, 138, 320.
__device__ __forceinline__ int32_t leaf_moments32_thread(
    int64_t b, TreeNode *node, Mom32 *m32, double *nrs, const float4 *spA, const float4 *spB,
    const float *sml, const double *srs, const int32_t *sq, const double *box,
    const SegView &sv) {
  {
    TreeNode *nd = &node[b];
    const int4 r2 = reinterpret_cast<const int4 *>(nd)[2], r3 = reinterpret_cast<const int4 *>(nd)[3];
    const int32_t f = r3.z, c = r3.w;
    const double L = box[5 * seg_at(sv, f) + 3];
    const float4 A0 = spA[f], B0 = spB[f];
    FF M{0.f, 0.f}, D[3] = {{0.f, 0.f}, {0.f, 0.f}, {0.f, 0.f}};
    float S[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    int64_t rsb = 0;
    int32_t lo[3] = {P3T_QMAX, P3T_QMAX, P3T_QMAX}, hi[3] = {-1, -1, -1};
    for (int32_t i = f; i < f + c; ++i) {
      const float4 A = spA[i], B = spB[i];
      const FF dx = ff_add({A.x, B.x}, {-A0.x, -B0.x});
      const FF dy = ff_add({A.y, B.y}, {-A0.y, -B0.y});
      const FF dz = ff_add({A.z, B.z}, {-A0.z, -B0.z});
      const FF m = ff_fast(A.w, sml[i]);
      M = ff_add(M, m);
      D[0] = ff_add(D[0], ff_mul(m, dx));
      D[1] = ff_add(D[1], ff_mul(m, dy));
      D[2] = ff_add(D[2], ff_mul(m, dz));
      const float mx = m.h * dx.h, my = m.h * dy.h, mz = m.h * dz.h;
      S[0] = fmaf(mx, dx.h, S[0]); S[1] = fmaf(my, dy.h, S[1]); S[2] = fmaf(mz, dz.h, S[2]);
      S[3] = fmaf(mx, dy.h, S[3]); S[4] = fmaf(mx, dz.h, S[4]); S[5] = fmaf(my, dz.h, S[5]);
      rsb = max_bits(rsb, srs[i]);
#pragma unroll
      for (int a = 0; a < 3; ++a) { lo[a] = min(lo[a], sq[3 * i + a]); hi[a] = max(hi[a], sq[3 * i + a]); }
    }
    const FF e[3] = {ff_div(D[0], M), ff_div(D[1], M), ff_div(D[2], M)};
    const FF cx = ff_add({A0.x, B0.x}, e[0]), cy = ff_add({A0.y, B0.y}, e[1]),
             cz = ff_add({A0.z, B0.z}, e[2]);
    const float Mh = M.h, ex = e[0].h, ey = e[1].h, ez = e[2].h;
    const float Cxx = S[0] - Mh * ex * ex, Cyy = S[1] - Mh * ey * ey, Czz = S[2] - Mh * ez * ez;
    const float tr = Cxx + Cyy + Czz;
    Mom32 o;
    o.hi = make_float4(cx.h, cy.h, cz.h, M.h);
    o.lo = make_float4(cx.l, cy.l, cz.l, M.l);
    o.q0 = make_float4(3.f * Cxx - tr, 3.f * Cyy - tr, 3.f * Czz - tr, 3.f * (S[3] - Mh * ex * ey));
    o.q1 = make_float4(3.f * (S[4] - Mh * ex * ez), 3.f * (S[5] - Mh * ey * ez), 0.f, 0.f);
    for (int a = 0; a < 3; ++a) { nd->qlo[a] = lo[a]; nd->qhi[a] = hi[a]; }
    const double rs = __longlong_as_double(rsb);
    nrs[b] = rs;
    nd->R = reach_cells(rs, L, cell_scale(L));
    m32[b] = o;
    return r2.w;
  }
}

constexpr int kLeavesByLanes = 4;  // leaves a warp up to which eight lanes take each
struct LeafTerms {
  float v[14][32];  // m (h, l), m d (h, l) x 3, m d rounded x 3, d x 3; a column a lane
};
template <class T>
__device__ __forceinline__ T grp_shfl(unsigned gm, T v, int src) {
  return __shfl_sync(gm, v, src, 8);
}
__device__ __forceinline__ FF grp_shfl(unsigned gm, FF v, int src) {
  return {__shfl_sync(gm, v.h, src, 8), __shfl_sync(gm, v.l, src, 8)};
}
__device__ __forceinline__ FF grp_xor(unsigned gm, FF v, int o) {
  return {__shfl_xor_sync(gm, v.h, o), __shfl_xor_sync(gm, v.l, o)};
}
// box and largest r_search over the group's lanes
__device__ __forceinline__ void grp_box(unsigned gm, int32_t (&lo)[3], int32_t (&hi)[3],
                                        int64_t &rsb) {
#pragma unroll
  for (int o = 4; o > 0; o >>= 1) {
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      lo[a] = min(lo[a], __shfl_xor_sync(gm, lo[a], o));
      hi[a] = max(hi[a], __shfl_xor_sync(gm, hi[a], o));
    }
    const int64_t r = __shfl_xor_sync(gm, rsb, o);
    rsb = r > rsb ? r : rsb;
  }
}
// the group writes a node: box, reach and largest r_search, moments
__device__ __forceinline__ void grp_store(int64_t b, int sub, TreeNode *node, Mom32 *m32,
                                          double *nrs, const int32_t (&lo)[3],
                                          const int32_t (&hi)[3], int level, int64_t rsb, double L,
                                          const Mom32 &o) {
  int4 *n4 = reinterpret_cast<int4 *>(&node[b]);
  const double rs = __longlong_as_double(rsb);
  if (sub == 0) m32[b].hi = o.hi;
  if (sub == 1) m32[b].lo = o.lo;
  if (sub == 2) m32[b].q0 = o.q0;
  if (sub == 3) m32[b].q1 = o.q1;
  if (sub == 4) n4[0] = make_int4(lo[0], lo[1], lo[2], reach_cells(rs, L, cell_scale(L)));
  if (sub == 5) n4[1] = make_int4(hi[0], hi[1], hi[2], level);
  if (sub == 6) nrs[b] = rs;
}

__device__ __forceinline__ int32_t leaf_moments32_lanes(
    int64_t b, unsigned gm, int sub, LeafTerms &T, TreeNode *node, Mom32 *m32, double *nrs,
    const float4 *spA, const float4 *spB, const float *sml, const double *srs, const int32_t *sq,
    const double *box, const SegView &sv) {
  const int col0 = (threadIdx.x & 31) - sub;
  const int4 *n4 = reinterpret_cast<const int4 *>(&node[b]);
  const int4 r1 = n4[1], r2 = n4[2], r3 = n4[3];
  const int32_t f = r3.z, c = r3.w;
  const double L = box[5 * seg_at(sv, f) + 3];
  const float4 A0 = spA[f], B0 = spB[f];
  // lanes 0-3: M, D; lanes 4-6: (Sxx, Sxy), (Syy, Sxz), (Szz, Syz)
  FF acc{0.f, 0.f};
  float s0 = 0.f, s1 = 0.f;
  const int k0 = sub == 4 ? 8 : (sub == 5 ? 9 : 10), l0 = sub == 4 ? 11 : (sub == 5 ? 12 : 13);
  const int k1 = sub == 6 ? 9 : 8, l1 = sub == 4 ? 12 : 13;
  int64_t rsb = 0;
  int32_t lo[3] = {P3T_QMAX, P3T_QMAX, P3T_QMAX}, hi[3] = {-1, -1, -1};
  for (int32_t base = 0; base < c; base += 8) {
    const int32_t i = f + base + sub;
    if (base + sub < c) {
      const float4 A = spA[i], B = spB[i];
      const FF dx = ff_add({A.x, B.x}, {-A0.x, -B0.x});
      const FF dy = ff_add({A.y, B.y}, {-A0.y, -B0.y});
      const FF dz = ff_add({A.z, B.z}, {-A0.z, -B0.z});
      const FF m = ff_fast(A.w, sml[i]);
      const FF tx = ff_mul(m, dx), ty = ff_mul(m, dy), tz = ff_mul(m, dz);
      const int l = col0 + sub;
      T.v[0][l] = m.h; T.v[1][l] = m.l;
      T.v[2][l] = tx.h; T.v[3][l] = tx.l;
      T.v[4][l] = ty.h; T.v[5][l] = ty.l;
      T.v[6][l] = tz.h; T.v[7][l] = tz.l;
      T.v[8][l] = m.h * dx.h; T.v[9][l] = m.h * dy.h; T.v[10][l] = m.h * dz.h;
      T.v[11][l] = dx.h; T.v[12][l] = dy.h; T.v[13][l] = dz.h;
      rsb = max_bits(rsb, srs[i]);
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        lo[a] = min(lo[a], sq[3 * i + a]);
        hi[a] = max(hi[a], sq[3 * i + a]);
      }
    }
    __syncwarp(gm);
    const int nb = min(8, c - base);
    if (sub < 4) {
      for (int j = 0; j < nb; ++j)
        acc = ff_add(acc, {T.v[2 * sub][col0 + j], T.v[2 * sub + 1][col0 + j]});
    } else if (sub < 7) {
      for (int j = 0; j < nb; ++j) {
        s0 = fmaf(T.v[k0][col0 + j], T.v[l0][col0 + j], s0);
        s1 = fmaf(T.v[k1][col0 + j], T.v[l1][col0 + j], s1);
      }
    }
    __syncwarp(gm);
  }
  grp_box(gm, lo, hi, rsb);
  const FF M = grp_shfl(gm, acc, 0);
  const FF D[3] = {grp_shfl(gm, acc, 1), grp_shfl(gm, acc, 2), grp_shfl(gm, acc, 3)};
  const float S[6] = {grp_shfl(gm, s0, 4), grp_shfl(gm, s0, 5), grp_shfl(gm, s0, 6),
                      grp_shfl(gm, s1, 4), grp_shfl(gm, s1, 5), grp_shfl(gm, s1, 6)};
  const FF e[3] = {ff_div(D[0], M), ff_div(D[1], M), ff_div(D[2], M)};
  const FF cx = ff_add({A0.x, B0.x}, e[0]), cy = ff_add({A0.y, B0.y}, e[1]),
           cz = ff_add({A0.z, B0.z}, e[2]);
  const float Mh = M.h, ex = e[0].h, ey = e[1].h, ez = e[2].h;
  const float Cxx = S[0] - Mh * ex * ex, Cyy = S[1] - Mh * ey * ey, Czz = S[2] - Mh * ez * ez;
  const float tr = Cxx + Cyy + Czz;
  Mom32 o;
  o.hi = make_float4(cx.h, cy.h, cz.h, M.h);
  o.lo = make_float4(cx.l, cy.l, cz.l, M.l);
  o.q0 = make_float4(3.f * Cxx - tr, 3.f * Cyy - tr, 3.f * Czz - tr, 3.f * (S[3] - Mh * ex * ey));
  o.q1 = make_float4(3.f * (S[4] - Mh * ex * ez), 3.f * (S[5] - Mh * ey * ez), 0.f, 0.f);
  grp_store(b, sub, node, m32, nrs, lo, hi, r1.w, rsb, L, o);
  return r2.w;
}

// One internal node of the mixed path from its children's Mom32 records, a
// child a lane, the eight slots added in the fixed pairwise tree ((s0 + s4) +
// (s2 + s6)) + ((s1 + s5) + (s3 + s7)), zero past the last child (adding zero
// to a normalised sum returns it); lane 0 holds the sums.  The children were
// written by other threads of the same launch: read through L2.
__device__ int32_t node_moments32(int64_t b, unsigned gm, int sub, TreeNode *node, Mom32 *m32,
                                  double *nrs, const double *box, const SegView &sv) {
  const int4 *n4 = reinterpret_cast<const int4 *>(&node[b]);
  const int4 r1 = __ldcg(n4 + 1), r2 = __ldcg(n4 + 2), r3 = __ldcg(n4 + 3);
  const int32_t c0 = r3.x, nch = r3.y;
  if (nch < 1 || nch > 8) return r2.w;  // only a node with children is completed
  int64_t rsb = 0;
  int32_t lo[3] = {P3T_QMAX, P3T_QMAX, P3T_QMAX}, hi[3] = {-1, -1, -1};
  const bool on = sub < nch;
  Mom32 cm;
  cm.hi = cm.lo = cm.q0 = cm.q1 = make_float4(0.f, 0.f, 0.f, 0.f);
  FF P[4] = {{0.f, 0.f}, {0.f, 0.f}, {0.f, 0.f}, {0.f, 0.f}};
  if (on) {
    const Mom32 *m = &m32[c0 + sub];
    cm.hi = __ldcg(&m->hi); cm.lo = __ldcg(&m->lo); cm.q0 = __ldcg(&m->q0); cm.q1 = __ldcg(&m->q1);
    const int4 *cn = reinterpret_cast<const int4 *>(&node[c0 + sub]);
    const int4 q0 = __ldcg(cn), q1 = __ldcg(cn + 1);
    rsb = max_bits(0, __ldcg(&nrs[c0 + sub]));
    lo[0] = q0.x; lo[1] = q0.y; lo[2] = q0.z;
    hi[0] = q1.x; hi[1] = q1.y; hi[2] = q1.z;
    P[0] = ff_fast(cm.hi.w, cm.lo.w);
    P[1] = ff_mul(P[0], ff_fast(cm.hi.x, cm.lo.x));
    P[2] = ff_mul(P[0], ff_fast(cm.hi.y, cm.lo.y));
    P[3] = ff_mul(P[0], ff_fast(cm.hi.z, cm.lo.z));
  }
  grp_box(gm, lo, hi, rsb);
#pragma unroll
  for (int o = 4; o > 0; o >>= 1)
#pragma unroll
    for (int q = 0; q < 4; ++q) P[q] = ff_add(P[q], grp_xor(gm, P[q], o));
#pragma unroll
  for (int q = 0; q < 4; ++q) P[q] = grp_shfl(gm, P[q], 0);
  const FF pc[3] = {ff_div(P[1], P[0]), ff_div(P[2], P[0]), ff_div(P[3], P[0])};
  float Q[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
  if (on) {
    const float M = cm.hi.w;
    const float dx = ff_add(ff_fast(cm.hi.x, cm.lo.x), ff_neg(pc[0])).h;
    const float dy = ff_add(ff_fast(cm.hi.y, cm.lo.y), ff_neg(pc[1])).h;
    const float dz = ff_add(ff_fast(cm.hi.z, cm.lo.z), ff_neg(pc[2])).h;
    const float d2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
    const float tx = 3.f * dx, ty = 3.f * dy;
    Q[0] = fmaf(M, fmaf(tx, dx, -d2), cm.q0.x);
    Q[1] = fmaf(M, fmaf(ty, dy, -d2), cm.q0.y);
    Q[2] = fmaf(M, fmaf(3.f * dz, dz, -d2), cm.q0.z);
    Q[3] = fmaf(M, tx * dy, cm.q0.w);
    Q[4] = fmaf(M, tx * dz, cm.q1.x);
    Q[5] = fmaf(M, ty * dz, cm.q1.y);
  }
#pragma unroll
  for (int o = 4; o > 0; o >>= 1)
#pragma unroll
    for (int q = 0; q < 6; ++q) Q[q] = Q[q] + __shfl_xor_sync(gm, Q[q], o);
  Mom32 o;
  o.hi = make_float4(pc[0].h, pc[1].h, pc[2].h, P[0].h);
  o.lo = make_float4(pc[0].l, pc[1].l, pc[2].l, P[0].l);
#pragma unroll
  for (int q = 0; q < 6; ++q) Q[q] = grp_shfl(gm, Q[q], 0);
  o.q0 = make_float4(Q[0], Q[1], Q[2], Q[3]);
  o.q1 = make_float4(Q[4], Q[5], 0.f, 0.f);
  grp_store(b, sub, node, m32, nrs, lo, hi, r1.w, rsb, box[5 * seg_at(sv, r3.z) + 3], o);
  return r2.w;
}

// the group writes an FP64 node's box, reach and largest r_search
__device__ __forceinline__ void grp_store64(int64_t b, int sub, TreeNode *node, double *nrs,
                                            const int32_t (&lo)[3], const int32_t (&hi)[3],
                                            int level, int64_t rsb, double L) {
  int4 *n4 = reinterpret_cast<int4 *>(&node[b]);
  const double rs = __longlong_as_double(rsb);
  if (sub == 3) n4[0] = make_int4(lo[0], lo[1], lo[2], reach_cells(rs, L, cell_scale(L)));
  if (sub == 7) n4[1] = make_int4(hi[0], hi[1], hi[2], level);
  if (sub == 1) nrs[b] = rs;
}

// An FP64 leaf by eight lanes: the members multiplied out one a lane, the ten
// sums (leaf_moments64_thread's, in the member order) dealt to the lanes: lane
// l the sum l of M, D, Sxx, Syy, Szz, Sxy, and by its parity Sxz or Syz
struct LeafTerms64 {
  double v[7][32];  // m, m d, d; a column a lane
};
__device__ __forceinline__ int32_t leaf_moments64_lanes(
    int64_t b, unsigned gm, int sub, LeafTerms64 &T, TreeNode *node, Mom64 *m64, double *nrs,
    const double *sx, const double *sy, const double *sz, const double *sm, const double *srs,
    const int32_t *sq, const double *box, const SegView &sv) {
  const int col0 = (threadIdx.x & 31) - sub;
  const int4 *n4 = reinterpret_cast<const int4 *>(&node[b]);
  const int4 r1 = n4[1], r2 = n4[2], r3 = n4[3];
  const int32_t f = r3.z, c = r3.w;
  const double L = box[5 * seg_at(sv, f) + 3];
  const double rx = sx[f], ry = sy[f], rz = sz[f];
  // the factors' rows of the lane's two sums (row k1 < 4: the factor is one)
  const int k0 = sub < 4 ? sub : (sub == 7 ? 1 : sub - 3), k1 = sub < 4 ? 0 : (sub == 7 ? 5 : sub);
  const int h0 = 1 + (sub & 1);
  double s0 = 0.0, s1 = 0.0;
  int64_t rsb = 0;
  int32_t lo[3] = {P3T_QMAX, P3T_QMAX, P3T_QMAX}, hi[3] = {-1, -1, -1};
  for (int32_t base = 0; base < c; base += 8) {
    const int32_t i = f + base + sub;
    if (base + sub < c) {
      const double m = sm[i], dx = sx[i] - rx, dy = sy[i] - ry, dz = sz[i] - rz;
      const int l = col0 + sub;
      T.v[0][l] = m;
      T.v[1][l] = m * dx; T.v[2][l] = m * dy; T.v[3][l] = m * dz;
      T.v[4][l] = dx; T.v[5][l] = dy; T.v[6][l] = dz;
      rsb = max_reach(rsb, srs[i]);
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        lo[a] = min(lo[a], sq[3 * i + a]);
        hi[a] = max(hi[a], sq[3 * i + a]);
      }
    }
    __syncwarp(gm);
    const int nb = min(8, c - base);
    for (int j = 0; j < nb; ++j) {
      const double w = T.v[k1][col0 + j];
      s0 = __fma_rn(T.v[k0][col0 + j], k1 < 4 ? 1.0 : w, s0);
      s1 = __fma_rn(T.v[h0][col0 + j], T.v[6][col0 + j], s1);
    }
    __syncwarp(gm);
  }
  grp_box(gm, lo, hi, rsb);
  const double M = grp_shfl(gm, s0, 0);
  const double iM = 1.0 / M;
  const double el = s0 * iM;  // lanes 1-3: e
  const double e[3] = {grp_shfl(gm, el, 1), grp_shfl(gm, el, 2), grp_shfl(gm, el, 3)};
  // lane 4 + q: C of xx, yy, zz, xy; lanes 0, 1: xz, yz
  const double ea = sub == 4 || sub == 7 || sub == 0 ? e[0] : (sub == 6 ? e[2] : e[1]);
  const double eb = sub == 4 ? e[0] : (sub == 5 || sub == 7 ? e[1] : e[2]);
  const double C = (sub >= 4 ? s0 : s1) - M * ea * eb;
  const double tr = grp_shfl(gm, C, 4) + grp_shfl(gm, C, 5) + grp_shfl(gm, C, 6);
  const double C3 = 3.0 * C, Q = C3 - tr;
  double *o = reinterpret_cast<double *>(&m64[b]);
  if (sub == 0) o[3] = M;
  if (sub >= 1 && sub < 4) o[sub - 1] = (sub == 1 ? rx : (sub == 2 ? ry : rz)) + el;
  if (sub >= 4) o[sub] = sub < 7 ? Q : C3;
  if (sub < 2) o[8 + sub] = C3;
  grp_store64(b, sub, node, nrs, lo, hi, r1.w, rsb, L);
  return r2.w;
}

// One step of the sum over the group's eight lanes: the lanes with the bit set
// keep the upper half of the values, the others the lower half, each added to
// the partner's (so that every value is added once a step, not in every lane)
template <int N>
__device__ __forceinline__ void halve(unsigned gm, bool up, int bit, double (&v)[N]) {
  constexpr int H = (N + 1) / 2;
#pragma unroll
  for (int q = 0; q < H; ++q) {
    const int u = q + N / 2;  // an odd middle value is kept by both
    const double keep = up ? v[u] : v[q], give = up ? v[q] : v[u];
    v[q] = keep + __shfl_xor_sync(gm, give, bit);
  }
}

// One internal node of the FP64 path, a child a lane, the eight slots (zero
// past the last child) added in the same fixed pairwise tree as the mixed
// path's
__device__ int32_t node_moments64(int64_t b, unsigned gm, int sub, TreeNode *node, Mom64 *m64,
                                  double *nrs, const double *box, const SegView &sv) {
  const int4 *n4 = reinterpret_cast<const int4 *>(&node[b]);
  const int4 r1 = __ldcg(n4 + 1), r2 = __ldcg(n4 + 2), r3 = __ldcg(n4 + 3);
  const int32_t c0 = r3.x, nch = r3.y;
  if (nch < 1 || nch > 8) return r2.w;  // only a node with children is completed
  int64_t rsb = 0;
  int32_t lo[3] = {P3T_QMAX, P3T_QMAX, P3T_QMAX}, hi[3] = {-1, -1, -1};
  const bool on = sub < nch;
  double2 g[5];
#pragma unroll
  for (int k = 0; k < 5; ++k) g[k] = make_double2(0.0, 0.0);
  if (on) {
    const double2 *m = reinterpret_cast<const double2 *>(&m64[c0 + sub]);
#pragma unroll
    for (int k = 0; k < 5; ++k) g[k] = __ldcg(m + k);
    const int4 *cn = reinterpret_cast<const int4 *>(&node[c0 + sub]);
    const int4 q0 = __ldcg(cn), q1 = __ldcg(cn + 1);
    rsb = max_bits(0, __ldcg(&nrs[c0 + sub]));
    lo[0] = q0.x; lo[1] = q0.y; lo[2] = q0.z;
    hi[0] = q1.x; hi[1] = q1.y; hi[2] = q1.z;
  }
  grp_box(gm, lo, hi, rsb);
  const double m = g[1].y;
  double t4[4] = {m, m * g[0].x, m * g[0].y, m * g[1].x};
  const bool b4 = sub & 4, b2 = sub & 2, b1 = sub & 1;
  halve(gm, b4, 4, t4);
  double t2[2] = {t4[0], t4[1]};
  halve(gm, b2, 2, t2);
  const double t = t2[0] + __shfl_xor_sync(gm, t2[0], 1);  // lane 2c: sum c of M, M com
  const double M = grp_shfl(gm, t, 0);
  const double iM = 1.0 / M;
  const double cl = t * iM;
  const double cx = grp_shfl(gm, cl, 2), cy = grp_shfl(gm, cl, 4), cz = grp_shfl(gm, cl, 6);
  double Q[6] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
  if (on) {
    const double dx = g[0].x - cx, dy = g[0].y - cy, dz = g[1].x - cz;
    const double d2 = __fma_rn(dx, dx, __fma_rn(dy, dy, dz * dz));
    const double tx = 3.0 * dx, ty = 3.0 * dy;
    Q[0] = __fma_rn(m, __fma_rn(tx, dx, -d2), g[2].x);
    Q[1] = __fma_rn(m, __fma_rn(ty, dy, -d2), g[2].y);
    Q[2] = __fma_rn(m, __fma_rn(3.0 * dz, dz, -d2), g[3].x);
    Q[3] = __fma_rn(m, tx * dy, g[3].y);
    Q[4] = __fma_rn(m, tx * dz, g[4].x);
    Q[5] = __fma_rn(m, ty * dz, g[4].y);
  }
  halve(gm, b4, 4, Q);
  double Q3[3] = {Q[0], Q[1], Q[2]};
  // three values: the lower lanes keep 0 and 1, the upper ones 2 (in [1])
  halve(gm, b2, 2, Q3);
  const double keep = b2 ? Q3[1] : (b1 ? Q3[1] : Q3[0]), give = b2 ? Q3[1] : (b1 ? Q3[0] : Q3[1]);
  const double q = keep + __shfl_xor_sync(gm, give, 1);
  double *o = reinterpret_cast<double *>(&m64[b]);
  if (sub == 0) o[3] = M;
  if (sub == 2) o[0] = cl;
  if (sub == 4) o[1] = cl;
  if (sub == 6) o[2] = cl;
  if ((sub & 3) != 3) o[4 + (b4 ? 3 : 0) + (sub & 3)] = q;
  grp_store64(b, sub, node, nrs, lo, hi, r1.w, rsb, box[5 * seg_at(sv, r3.z) + 3]);
  return r2.w;
}

// All moments in one launch, bottom-up: a leaf, once computed, is counted off
// at its parent (node_done, preset to the number of children by k_nodes_bfs);
// the child that brings the count to zero makes the parent ready, which its
// warp takes next, four nodes at a time (each node's record gives its parent
// in the same load as its children).  Nothing waits, and a node's result does
// not depend on which child arrives last.
struct MomArgs {
  const int64_t *nleaf;
  const int32_t *leaf_list;
  TreeNode *node;
  Mom32 *m32;
  Mom64 *m64;
  double *nrs;
  const float4 *spA, *spB;
  const float *sml;
  const double *sx, *sy, *sz, *sm, *srs;
  const int32_t *sq;
  const double *box;
  SegView sv;
  int32_t *node_done;
};
template <bool MIXED> struct MomTerms { using type = LeafTerms; };
template <> struct MomTerms<false> { using type = LeafTerms64; };
template <bool MIXED>
__global__ void __launch_bounds__(128) k_moments_up(MomArgs g) {
  pdl_wait();
  __shared__ typename MomTerms<MIXED>::type s_t[4];
  __shared__ int32_t s_ready[4][32];
  const int64_t nleaf = *g.nleaf;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, sub = lane & 7, grp = lane >> 3;
  const unsigned gm = 0xffu << (lane & 24), lt = (1u << lane) - 1u;
  int32_t *ready = s_ready[w];
  const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  const int64_t warp = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const bool lanes = nleaf <= nwarps * kLeavesByLanes;  // leaves a warp takes at once
  const int per = lanes ? 4 : 32;
  for (int64_t t0 = warp * per; t0 < nleaf; t0 += nwarps * per) {
    const int64_t t = t0 + (lanes ? grp : lane);
    int32_t p = -1;  // held by one lane a leaf
    if (lanes) {
      if (t < nleaf) {
        const int32_t b = g.leaf_list[t];
        if constexpr (MIXED)
          p = leaf_moments32_lanes(b, gm, sub, s_t[w], g.node, g.m32, g.nrs, g.spA, g.spB, g.sml,
                                   g.srs, g.sq, g.box, g.sv);
        else
          p = leaf_moments64_lanes(b, gm, sub, s_t[w], g.node, g.m64, g.nrs, g.sx, g.sy, g.sz,
                                   g.sm, g.srs, g.sq, g.box, g.sv);
        if (sub != 0) p = -1;
      }
    } else if (t < nleaf) {
      const int32_t b = g.leaf_list[t];
      if constexpr (MIXED)
        p = leaf_moments32_thread(b, g.node, g.m32, g.nrs, g.spA, g.spB, g.sml, g.srs, g.sq, g.box,
                                  g.sv);
      else
        p = leaf_moments64_thread(b, g.node, g.m64, g.nrs, g.sx, g.sy, g.sz, g.sm, g.srs, g.sq,
                                  g.box, g.sv);
    }
    int n = 0;  // nodes ready, all of their children done
    for (;;) {
      __threadfence();  // the nodes' records before the counts
      __syncwarp();
      const bool last = p >= 0 && atomicSub(&g.node_done[p], 1) == 1;
      const unsigned m = __ballot_sync(0xffffffffu, last);
      if (last) ready[n + __popc(m & lt)] = p;
      n += __popc(m);
      __syncwarp();
      if (n == 0) break;
      __threadfence();  // the siblings' records after their counts
      const int take = n < 4 ? n : 4;
      const int32_t b = grp < take ? ready[n - 1 - grp] : -1;
      n -= take;
      __syncwarp();
      p = -1;
      if (b >= 0) {
        if constexpr (MIXED)
          p = node_moments32(b, gm, sub, g.node, g.m32, g.nrs, g.box, g.sv);
        else
          p = node_moments64(b, gm, sub, g.node, g.m64, g.nrs, g.box, g.sv);
        if (sub != 0) p = -1;
      }
    }
  }
}

__global__ void k_tree_stats(const int64_t *d_nnode, int64_t node_cap,
                             const TreeNode *node, int64_t *stats) {
  pdl_wait();
  const int64_t nn = min(*d_nnode, node_cap);
  unsigned long long depth = 0, maxleaf = 0, nleaf = 0;
  for (int64_t b = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; b < nn;
       b += (int64_t)gridDim.x * blockDim.x) {
    depth = max(depth, (unsigned long long)node[b].level);
    if (node[b].nchild == 0) { ++nleaf; maxleaf = max(maxleaf, (unsigned long long)node[b].count); }
  }
  for (int o = 16; o > 0; o >>= 1) {
    depth = max(depth, __shfl_xor_sync(0xffffffffu, depth, o));
    maxleaf = max(maxleaf, __shfl_xor_sync(0xffffffffu, maxleaf, o));
    nleaf += __shfl_xor_sync(0xffffffffu, nleaf, o);
  }
  if ((threadIdx.x & 31) == 0) {
    atomicMax(reinterpret_cast<unsigned long long *>(&stats[2]), depth);
    atomicMax(reinterpret_cast<unsigned long long *>(&stats[3]), maxleaf);
    atomicAdd(reinterpret_cast<unsigned long long *>(&stats[1]), nleaf);
  }
}

}  // namespace

// counters layout (int64): [0] n, [1] nodes, [2] leaves, [3] nodes clamped to
// the capacity, [4..7] tree stats, [8] candidates, [9] candidates clamped,
// [10] neighbour entries, [11] cluster members, [12] walk group cursor
// radial bins of a system of n particles (Sec. 2.1.3 reading C3)
static int cut_bins(int vran_bins, int64_t n) {
  int nb = vran_bins;
  if (nb <= 0) { int64_t t = n / 1000; nb = (int)(t < 1 ? 1 : (t > 1024 ? 1024 : t)); }
  return nb;
}

// slices a segment for a reduction over every segment, none with less than a
// trip of a block (four elements a thread): of one system a few blocks per SM
// in all, of several as many as the longest one asks for (two slices a segment
// of 518 to 16,296 particles: 60 us for the root cubes, 27 now)
static int box_slices(const p3t_ctx *c, int64_t n) {
  const int64_t most = c->nseg == 1 ? 4 * c->num_sms : p3t_box_blocks(c->num_sms) / c->nseg;
  const int64_t len = c->nseg == 1 ? n : c->seg_max;
  return (int)std::min(most, (len + 4 * kBlock - 1) / (4 * kBlock) + 1);
}

int p3t_run_cutoffs(p3t_ctx *c, p3t_particles *p, cudaStream_t s) {
  const int64_t n = p->n;
  if (n == 0) return P3T_OK;
  const SegView sv{c->seg_off, (int)c->nseg, n};
  int64_t nbt = 0;  // bins of all segments
  if (c->nseg == 1) {
    nbt = cut_bins(c->prm.vran_bins, n);
  } else {
    for (int64_t d = 0; d < c->nseg; ++d)
      nbt += cut_bins(c->prm.vran_bins, c->seg_off_h[d + 1] - c->seg_off_h[d]);
  }
  if (nbt > kMaxBins) return P3T_ERR_INVALID;
  const int nb = (int)nbt;
  double *bsum = c->epart;  // reuse: >= 4096 doubles
  const int64_t g = p3t_grid(n, kBlock, (int64_t)c->num_sms * P3T_NSM_BLOCKS);
  int64_t *d_n = &c->counters[18];
  const int rsl = box_slices(c, n);
  pdl_launch(k_cut_range, dim3((unsigned)(rsl * c->nseg)), dim3(kBlock), 0, s, sv, rsl, p->x, p->y,
             c->box_part, c->seg_done, c->box_bits, nb, d_n);
  if (c->nseg > 1)
    pdl_launch(k_cut_segbins, dim3(1), dim3(1024), 0, s, sv, c->prm.vran_bins, c->box_bits, c->seg_nb,
                                     c->seg_base, c->seg_l);
  const double mu = c->prm.G * c->prm.m_star;
  // per-bin sums in a fixed order (particles grouped by bin with the stable
  // radix sort, then one warp per bin): the radii do not depend on timing
  double *u2 = c->hw;
  int32_t *bin = c->flag;  // the bins of k_cut_u2, read by k_cut_final (N int32)
  pdl_launch(k_cut_u2, dim3((unsigned)g), dim3(kBlock), 0, s, sv, p->x, p->y, p->z, p->vx, p->vy, p->vz, sqrt(mu),
                                          c->box_bits, nb, c->seg_nb, c->seg_base, c->seg_l,
                                          u2, c->keys, c->idx, bin);
  int rc = p3t_sort_pairs(&c->keys, &c->idx, &c->keys_alt, &c->idx_alt, d_n, c->cap, nb <= 256 ? 8 : 16,
                          c->radix_hist, c->radix_hist_cap, c->sort_work, p3t_sort_where(c), s);
  if (rc) return rc;
  pdl_launch(k_cut_binsum, dim3((unsigned)p3t_grid((int64_t)nb * 32, kBlock, (int64_t)c->num_sms * 4)),
             dim3(kBlock), 0, s, nb, n, c->keys, c->idx, u2, bsum);
  pdl_launch(k_cut_final, dim3((unsigned)g), dim3(kBlock), 0, s, sv, p->x, p->y, p->z, p->vx, p->vy,
                                             p->vz, p->m, c->prm, 1.0 / mu,
                                             1.0 / (3.0 * c->prm.m_star), c->box_bits, bin, bsum,
                                             p->r_out, p->r_search);
  if (c->prm.cutoff_mode == P3T_CUT_SHARED)
    pdl_launch(k_cut_shared, dim3((unsigned)g), dim3(kBlock), 0, s, sv, c->box_bits, p->r_out, p->r_search);
  // range, u2, bin sums, final (+ shared, + segment bins); the sort counts
  // itself
  p3t_note_launches(4 + (c->prm.cutoff_mode == P3T_CUT_SHARED) + (c->nseg > 1));
  return cudaGetLastError() == cudaSuccess ? P3T_OK : P3T_ERR_CUDA;
}

int p3t_run_build_tree(p3t_ctx *c, const p3t_particles *p, cudaStream_t s) {
  const int64_t n = p->n;
  const int leaf = c->prm.leaf_size;
  const int64_t maxb = (int64_t)c->num_sms * P3T_NSM_BLOCKS;
  const int64_t g = p3t_grid(n, kBlock, maxb);
  int64_t *cnt = c->counters;
  int rc;
  const int nseg = (int)c->nseg;
  const SegView sv{c->seg_off, nseg, n};
  const int bsl = box_slices(c, n);
  pdl_launch(k_box, dim3((unsigned)(bsl * nseg)), dim3(kBlock), 0, s, sv, bsl, p->x, p->y, p->z,
             c->box_part, c->seg_done, c->box);
  pdl_launch(k_keys, dim3((unsigned)g), dim3(kBlock), 0, s, sv, p->x, p->y, p->z, p->m, p->r_out, p->r_search,
                                        c->box, c->keys, c->idx, c->pack, 0, &cnt[0]);
  // several systems of which none is above P3T_SORT_SEGMENT are sorted apart: 256
  // disks of 518 to 16,296 particles 99 us of kernels, one sort of all with a
  // pass by segment and the keys anew 204.  Above, a segment's merges would be
  // more rounds over memory than the one sort's passes
  const bool apart = nseg > 1 && c->seg_max <= P3T_SORT_SEGMENT;
  if (apart)
    rc = p3t_sort_segments(sv, c->keys, c->idx, c->keys_alt, c->idx_alt, c->seg_max, c->cap, 63,
                           s);
  else
    rc = p3t_sort_pairs(&c->keys, &c->idx, &c->keys_alt, &c->idx_alt, &cnt[0], c->cap, 63,
                        c->radix_hist, c->radix_hist_cap, c->sort_work, p3t_sort_where(c), s);
  if (rc) return rc;
  if (nseg > 1 && !apart) {
    // stable sort by segment (the most significant digit of (segment, key)),
    // then the keys of the new order
    int sbits = 0;
    while ((1 << sbits) < nseg) ++sbits;
    pdl_launch(k_segkey, dim3((unsigned)g), dim3(kBlock), 0, s, sv, c->idx, c->keys);
    rc = p3t_radix_sort(&c->keys, &c->idx, &c->keys_alt, &c->idx_alt, &cnt[0], c->cap,
                        0, sbits, c->radix_hist, c->radix_hist_cap, s);
    if (rc) return rc;
    pdl_launch(k_keys, dim3((unsigned)g), dim3(kBlock), 0, s, sv, p->x, p->y, p->z, p->m, p->r_out, p->r_search,
                                          c->box, c->keys, c->idx, c->pack, 1, nullptr);
    p3t_note_launches(2);
  }
  auto gather = c->prm.precision == P3T_MIXED ? k_gather<true> : k_gather<false>;
  pdl_launch(gather, dim3((unsigned)p3t_grid(n, kLevelTile, maxb)), dim3(kLevelTile), 0, s, sv,
             c->idx, c->keys, c->pack, c->sx, c->sy, c->sz, c->sm, c->sro, c->srs, c->sq, c->spA,
             c->spB, c->srs32, c->sml, leaf, c->lp, c->lv, c->ncount);
  rc = p3t_scan_i32_to_i64(c->ncount, c->nstart, &cnt[0], c->cap, &cnt[1], c->scan_state, c->scan_words, c->status, c->poll_limit, s);
  if (rc) return rc;
  pdl_launch(k_nodes_pre, dim3((unsigned)g), dim3(kBlock), 0, s, sv, c->lp, c->lv, c->nstart, cnt, c->node_cap,
                                             c->pre_first, c->pre_level, c->lvl_keys,
                                             c->bfs2pre, c->status);
  pdl_launch(k_node_counts, dim3((unsigned)p3t_grid(c->node_cap, kBlock, maxb)), dim3(kBlock), 0, s, 
      sv, c->keys, &cnt[1], c->node_cap, c->pre_first, c->pre_level, c->pre_count, c->status);
  // breadth-first order: one block's counts, or a radix pass on the level that
  // also writes the inverse.  One block's time grows with the nodes, three
  // launches cost about the same at any size (whole tree build, block / pass: N
  // = 1,000 58 / 63 us, 3,001 71 / 75, 4,800, near the limit, 79 / 82)
  if (c->node_cap <= kOrderMax) {
    pdl_launch(k_level_order, dim3(1), dim3(1024), 0, s, &cnt[3], c->pre_level, c->bfs2pre,
               c->pre2bfs);
    p3t_note_launches(1);
  } else {
    rc = p3t_radix_sort(&c->lvl_keys, &c->bfs2pre, &c->lvl_keys_alt, &c->bfs2pre_alt, &cnt[3],
                        c->node_cap, 0, 8, c->radix_hist, c->radix_hist_cap, s, c->pre2bfs);
    if (rc) return rc;
  }
  const int64_t gn = p3t_grid(c->node_cap, kBlock, maxb);
  pdl_launch(k_nodes_bfs, dim3((unsigned)gn), dim3(kBlock), 0, s, &cnt[3], c->node_cap, c->bfs2pre, c->pre2bfs,
                                              c->pre_first, c->pre_count, c->pre_level,
                                              c->lp, c->lv, c->nstart, c->sq, c->node,
                                              c->prm.group_size, c->node_flag, c->node_done,
                                              c->status);
  // leaves (bit 0) and target groups (bit 1) counted by one scan
  rc = p3t_scan_flag_pairs(c->node_flag, c->flag_pos, &cnt[3], c->node_cap, &cnt[19],
                           c->scan_state, c->scan_words, c->status, c->poll_limit, s);
  if (rc) return rc;
  pdl_launch(k_lists, dim3((unsigned)gn), dim3(kBlock), 0, s, &cnt[3], c->node_cap, c->node_flag,
             c->flag_pos, c->pre2bfs, &cnt[19], c->leaf_list, c->group_list, &cnt[2], &cnt[15]);
  const MomArgs ma{&cnt[2], c->leaf_list, c->node, c->mom32, c->mom64, c->nrs, c->spA, c->spB,
                   c->sml, c->sx, c->sy, c->sz, c->sm, c->srs, c->sq, c->box, sv, c->node_done};
  auto moments = c->prm.precision == P3T_MIXED ? k_moments_up<true> : k_moments_up<false>;
  pdl_launch(moments, dim3((unsigned)p3t_grid(c->node_cap * 8, 128, maxb)), dim3(128), 0, s, ma);
  // own kernels here (the scans and sorts count themselves): box, keys, gather,
  // nodes_pre, node_counts, nodes_bfs, lists, moments
  p3t_note_launches(8);
  return cudaGetLastError() == cudaSuccess ? P3T_OK : P3T_ERR_CUDA;
}

// tree statistics on demand (diagnostics; not part of the step)
int p3t_run_tree_stats(p3t_ctx *c, cudaStream_t s) {
  int64_t *cnt = c->counters;
  P3T_CUDA_TRY(cudaMemsetAsync(&cnt[4], 0, 4 * sizeof(int64_t), s));
  const int64_t gn = p3t_grid(c->node_cap, kBlock, (int64_t)c->num_sms * P3T_NSM_BLOCKS);
  pdl_launch(k_tree_stats, dim3((unsigned)gn), dim3(kBlock), 0, s, &cnt[3], c->node_cap, c->node, &cnt[4]);
  p3t_note_launches(1);
  return cudaGetLastError() == cudaSuccess ? P3T_OK : P3T_ERR_CUDA;
}
