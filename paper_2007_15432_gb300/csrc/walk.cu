// Soft step: the changeover tree walk (Eq. softforce).
//
// One warp per target group (the highest tree node holding <= group_size
// particles, or a leaf), 32 targets per walk (larger groups are taken 32
// targets at a time; the warps take a group's first 32 targets and its rest
// as separate units of work, each walking with the whole group's box).  A walk
// of k < 32 targets gives each target r = floor(32 / k) lanes, each of which takes every r-th entry of a batch; the
// r partial sums are added at the end, so that lanes are not left idle.  The
// walk pops up to 32 nodes at a time from a per-warp stack, decides opening
// for all of them at once on the integer grid, and compacts accepted nodes,
// opened leaves and children with warp ballots / scans into shared-memory
// lists.  Each batch of 32 list entries is staged into shared memory once
// (one coalesced load per lane) and then read by every lane as a broadcast.
// Targets whose FP32 sum is ill-conditioned are redone in float-float right
// after their walk, all of them on one more traversal of the same list.
//
// Mixed path: positions are float-float (hi + lo) pairs, so a relative
// coordinate (x_i,hi - x_j,hi) + (x_i,lo - x_j,lo) carries the accuracy of an
// FP64 subtraction rounded to FP32, with no FP64 instruction per pair.  Pair
// and quadrupole terms are FP32; each batch's FP32 sum is folded into a
// float-float accumulator.  The mixed evaluators take the entries of a batch
// two at a time with packed FP32 pair instructions (add/sub/mul/fma.f32x2:
// one issue for two lanes' worth of FP32 work per thread), the batch staged
// so that one 16-byte shared load gives one coordinate of both entries;
// replicas split a batch by pairs, and each pair slot keeps its own partial
// sum (even and odd entries) until the batch is folded.  The FP64 path
// (k_walk64) shares the traversal and has a layout of its own.
#include <algorithm>

#include "p3t_internal.cuh"

namespace {

constexpr int kWarps = 4;                 // warps per block
constexpr int kPPCap = 32 * 33;           // p-p list: leftover < 32 + 32 leaves x <= 32
constexpr int kNDCap = 64;                // node list: leftover < 32 + 32 nodes
constexpr int kBigCap = 8;                // opened leaves with more than 32 members
// the FP32 candidate test r^2 < r_search^2 is widened by a factor 1.00001
// (applied to the squared radii in the gather); the exact FP64 test follows

struct WalkArgs {
  const TreeNode *node;
  const Mom64 *mom64;
  const Mom32 *mom32;
  const int32_t *leaf_list;
  const int64_t *d_nleaf;
  const int64_t *d_nnode;
  const double *sx, *sy, *sz, *sm, *sro, *srs;
  const float4 *spA, *spB;
  const float *srs32;
  const float *sml;          // mass lo parts (float-float masses with spA.w)
  const int32_t *idx;        // sorted -> caller
  double *ax, *ay, *az;      // caller order
  int32_t *stack;
  int64_t stack_cap;
  int32_t *cand_i, *cand_j;
  int64_t cand_cap;
  unsigned long long *cand_count;
  unsigned long long *counts;  // [2] n_pp, n_pnode (may be null)
  int64_t *cursor;
  DevStatus *st;
  SegView seg;                     // segments: the root of segment d is node d
  int group_max;                   // largest target group but for oversized leaves
  double G, gamma;
  double inv1mg;                   // 1 / (1 - gamma)
  float inv1mg_f, mgi_f;           // 1 / (1 - gamma), -gamma / (1 - gamma)
  float refine_cf;                 // refine when sum|term| > refine_cf * |a|
  int64_t bh[P3T_BITS + 1];
};

// integer box of a target group (a leaf) on the key grid
struct GroupBox {
  int32_t qlo0, qlo1, qlo2, qhi0, qhi1, qhi2, R;
  __device__ void load(const TreeNode &G) {
    qlo0 = G.qlo[0]; qlo1 = G.qlo[1]; qlo2 = G.qlo[2];
    qhi0 = G.qhi[0]; qhi1 = G.qhi[1]; qhi2 = G.qhi[2];
    R = G.R;
  }
};

__device__ __forceinline__ int warp_excl_scan(int v, int *total) {
  const int lane = threadIdx.x & 31;
  int x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    int t = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += t;
  }
  *total = __shfl_sync(0xffffffffu, x, 31);
  return x - v;
}

__device__ __forceinline__ void two_sum(float &hi, float &lo, float b) {
  const float s = hi + b;
  const float bb = s - hi;
  const float err = (hi - (s - bb)) + (b - bb);
  hi = s;
  lo += err;
}

// ---- per-target state (one lane per target) ---------------------------------
struct Target {
  f2 X, Y, Z, XL, YL, ZL;              // (hi, hi) and (lo, lo) of each coordinate
  float inv_ro, rs2;                   // rs2: r_search^2 with the FP32 margin
  float ahx, ahy, ahz, alx, aly, alz;  // float-float accumulators
  float tabs;                          // sum of term magnitudes (conditioning)
  int32_t self;
  int rep, nrep;                       // this lane's replica of the target, replicas
  bool valid;
  __device__ void load(const WalkArgs &a, int32_t ti, bool v, int r, int nr) {
    valid = v;
    self = ti;
    rep = r;
    nrep = nr;
    ahx = ahy = ahz = alx = aly = alz = 0.f;
    tabs = 0.f;
    if (v) {
      const float4 A = a.spA[ti], B = a.spB[ti];
      X = f2_dup(A.x); Y = f2_dup(A.y); Z = f2_dup(A.z);
      XL = f2_dup(B.x); YL = f2_dup(B.y); ZL = f2_dup(B.z);
      inv_ro = B.w;
      rs2 = a.srs32[ti];
    } else {  // far away: no force, no candidate
      X = Y = Z = f2_dup(3.0e30f);
      XL = YL = ZL = 0ull;
      inv_ro = 0.f;
      rs2 = 0.f;
    }
  }
  __device__ void fold(float bx, float by, float bz) {
    two_sum(ahx, alx, bx); two_sum(ahy, aly, by); two_sum(ahz, alz, bz);
  }
  // adds the partial sums of the other replicas (lanes lane + q k) into the
  // first; nrep and k are warp-uniform
  __device__ void reduce(int k) {
    const int lane = threadIdx.x & 31;
    for (int q = 1; q < nrep; ++q) {
      const int src = lane < k ? lane + q * k : lane;
      const float hx = __shfl_sync(0xffffffffu, ahx, src), lx = __shfl_sync(0xffffffffu, alx, src);
      const float hy = __shfl_sync(0xffffffffu, ahy, src), ly = __shfl_sync(0xffffffffu, aly, src);
      const float hz = __shfl_sync(0xffffffffu, ahz, src), lz = __shfl_sync(0xffffffffu, alz, src);
      const float tb = __shfl_sync(0xffffffffu, tabs, src);
      if (lane < k) {
        two_sum(ahx, alx, hx); alx += lx;
        two_sum(ahy, aly, hy); aly += ly;
        two_sum(ahz, alz, hz); alz += lz;
        tabs += tb;
      }
    }
  }
};

__device__ __forceinline__ void record_candidate(const WalkArgs &a, int32_t i,
                                                 int32_t j) {
  const unsigned long long slot = atomicAdd(a.cand_count, 1ull);
  if (slot < (unsigned long long)a.cand_cap) {
    a.cand_i[slot] = i;
    a.cand_j[slot] = j;
  }
}

// per-warp staging area for one batch of 32 entries
constexpr int kStageBytes = 32 * 96;
// mixed p-p batch by entry pairs (2p, 2p + 1): each 16-byte word holds one
// component of both entries, e.g. axy[p] = (x_2p, x_2p+1, y_2p, y_2p+1) of
// the hi parts; azw: z and mass; bxy, bzw: lo parts and 1 / r_out
struct StagePP32 {
  ulonglong2 axy[16], azw[16], bxy[16], bzw[16];
  float rs[32];
  int32_t idx[32];
};
// mixed node batch by pairs: centre hi / lo, -M, and the quadrupole
// (q0xy: xx, yy; q0zw: zz, xy; q1xy: xz, yz)
struct StageND32 {
  ulonglong2 hxy[16], hzw[16], lxy[16], lzw[16], q0xy[16], q0zw[16], q1xy[16];
};
static_assert(sizeof(StagePP32) <= kStageBytes && sizeof(StageND32) <= kStageBytes,
              "stage area");

// entry s of a pair-staged batch: component c (0..3) of word w
__device__ __forceinline__ void stage_put(ulonglong2 *w, int s, float v0, float v1) {
  float *f = reinterpret_cast<float *>(&w[s >> 1]);
  f[s & 1] = v0;
  f[2 + (s & 1)] = v1;
}

// ---- particle-particle batch ----------------------------------------------
// Changeover pair terms in FP32 on float-float relative coordinates, for the
// two entries of pair slot p at once.  r^2 is kept above 1e-30 for the
// reciprocal square root: a coincident pair (the target itself) has y = 0 <
// gamma, K = 0 and so adds nothing, and f is formed as ((m K) r^-1) r^-2 so
// that no factor overflows.  The candidate test compares r^2 with
// max(r_search^2) (squared and widened in the gather); far-away dummy targets
// and the massless dummy entry that pads an odd batch never pass it.  The
// batch sums are kept negated (B = -sum f dx), which is exact.
__device__ __forceinline__ void pp_pair(const WalkArgs &a, Target &t,
                                        const StagePP32 &S, int p, f2 &BX, f2 &BY, f2 &BZ,
                                        f2 &TB, unsigned &npp) {
  const ulonglong2 axy = S.axy[p], azw = S.azw[p], bxy = S.bxy[p], bzw = S.bzw[p];
  const f2 dx = add2(sub2(t.X, axy.x), sub2(t.XL, bxy.x));
  const f2 dy = add2(sub2(t.Y, axy.y), sub2(t.YL, bxy.y));
  const f2 dz = add2(sub2(t.Z, azw.x), sub2(t.ZL, bzw.x));
  const f2 r2 = fma2(dx, dx, fma2(dy, dy, mul2(dz, dz)));
  const float r2a = f2_lo(r2), r2b = f2_hi(r2);
  const f2 rinv = f2_pk(rsqrt_normal(fmaxf(r2a, 1e-30f)), rsqrt_normal(fmaxf(r2b, 1e-30f)));
  const f2 r = mul2(r2, rinv);
  const float ya = f2_lo(r) * fminf(t.inv_ro, f2_lo(bzw.y));
  const float yb = f2_hi(r) * fminf(t.inv_ro, f2_hi(bzw.y));
  const f2 x = f2_pk(__saturatef(fmaf(ya, a.inv1mg_f, a.mgi_f)),
                     __saturatef(fmaf(yb, a.inv1mg_f, a.mgi_f)));
  const f2 x2 = mul2(x, x);
  const f2 poly = fma2(fma2(fma2(f2_dup(-20.f), x, f2_dup(70.f)), x, f2_dup(-84.f)), x,
                       f2_dup(35.f));
  const f2 K = mul2(mul2(x2, x2), poly);
  const f2 f = mul2(mul2(mul2(azw.y, K), rinv), mul2(rinv, rinv));
  BX = fma2(f, dx, BX);
  BY = fma2(f, dy, BY);
  BZ = fma2(f, dz, BZ);
  TB = fma2(f, r, TB);
  if (r2a < fmaxf(t.rs2, S.rs[2 * p])) {
    const int32_t j = S.idx[2 * p];
    if (j != t.self) record_candidate(a, t.self, j);
    else --npp;  // the target itself is not a pair
  }
  if (r2b < fmaxf(t.rs2, S.rs[2 * p + 1])) {
    const int32_t j = S.idx[2 * p + 1];
    if (j != t.self) record_candidate(a, t.self, j);
    else --npp;
  }
}

// The targets' bounding box of one walk (float), the largest max(r_search^2,
// r_out^2) of its targets (widened like the candidate test) and the largest
// coordinate magnitude; per warp, in shared memory.
struct FarBox {
  float lo[3], hi[3], R2, amax;
};

// A source is far from every target of the walk when its distance to the
// box, less a margin that covers the FP32 rounding of the coordinates, is
// beyond max(r_search, r_out) of the source and of every target: then K = 1
// for every pair (y >= 1) and no pair is a neighbour candidate.
__device__ __forceinline__ bool far_from(const FarBox &b, const float4 A, const float4 B,
                                         float rs2s) {
  const float x = A.x + B.x, y = A.y + B.y, z = A.z + B.z;
  const float m = 9.5367431640625e-7f *  // 2^-20 of the coordinates' scale
                  (b.amax + fmaxf(fabsf(x), fmaxf(fabsf(y), fabsf(z))));
  const float gx = fmaxf(fmaxf(b.lo[0] - x, x - b.hi[0]) - m, 0.f);
  const float gy = fmaxf(fmaxf(b.lo[1] - y, y - b.hi[1]) - m, 0.f);
  const float gz = fmaxf(fmaxf(b.lo[2] - z, z - b.hi[2]) - m, 0.f);
  const float d2 = gx * gx + gy * gy + gz * gz;
  const float ro = 1.0f / B.w;  // B.w = 1 / r_out
  const float R2 = fmaxf(b.R2, fmaxf(rs2s, ro * ro * 1.00001f));
  return d2 > 0.f && d2 >= R2;
}

// pair terms with K = 1 and no candidate test (the batch is far, see above):
// the same operations as pp_pair's K = 1 case, so the same bits
__device__ __forceinline__ void pp_pair_far(Target &t, const StagePP32 &S, int p, f2 &BX,
                                            f2 &BY, f2 &BZ, f2 &TB) {
  const ulonglong2 axy = S.axy[p], azw = S.azw[p], bxy = S.bxy[p], bzw = S.bzw[p];
  const f2 dx = add2(sub2(t.X, axy.x), sub2(t.XL, bxy.x));
  const f2 dy = add2(sub2(t.Y, axy.y), sub2(t.YL, bxy.y));
  const f2 dz = add2(sub2(t.Z, azw.x), sub2(t.ZL, bzw.x));
  const f2 r2 = fma2(dx, dx, fma2(dy, dy, mul2(dz, dz)));
  const f2 rinv = f2_pk(rsqrt_normal(f2_lo(r2)), rsqrt_normal(f2_hi(r2)));
  const f2 r = mul2(r2, rinv);
  const f2 f = mul2(mul2(azw.y, rinv), mul2(rinv, rinv));
  BX = fma2(f, dx, BX);
  BY = fma2(f, dy, BY);
  BZ = fma2(f, dz, BZ);
  TB = fma2(f, r, TB);
}

// the batch sums of the even and odd slots into the target: the force sums
// negated back (B = -sum), the magnitude sum as it is
__device__ __forceinline__ void fold_pairs(Target &t, f2 BX, f2 BY, f2 BZ, f2 TB) {
  t.fold(-(f2_lo(BX) + f2_hi(BX)), -(f2_lo(BY) + f2_hi(BY)), -(f2_lo(BZ) + f2_hi(BZ)));
  t.tabs += f2_lo(TB) + f2_hi(TB);
}

template <int U>
__device__ __forceinline__ void eval_pp(const WalkArgs &a, Target &t, const int32_t *list,
                                        int nsrc, void *stage, const FarBox &box,
                                        unsigned &npp) {
  StagePP32 &S = *reinterpret_cast<StagePP32 *>(stage);
  const int lane = threadIdx.x & 31;
  bool near = false;
  float4 A = make_float4(1.0e18f, 1.0e18f, 1.0e18f, 0.f), B = make_float4(0.f, 0.f, 0.f, 0.f);
  float rs = 0.f;
  int32_t j = -1;
  if (lane < nsrc) {
    j = list[lane];
    A = __ldg(&a.spA[j]);
    B = __ldg(&a.spB[j]);
    rs = __ldg(&a.srs32[j]);
    near = !far_from(box, A, B, rs);
  }
  // lanes past the batch stage a massless dummy far from everything
  stage_put(S.axy, lane, A.x, A.y);
  stage_put(S.azw, lane, A.z, A.w);
  stage_put(S.bxy, lane, B.x, B.y);
  stage_put(S.bzw, lane, B.z, B.w);
  S.rs[lane] = rs;
  S.idx[lane] = j;
  const bool any_near = __any_sync(0xffffffffu, near);
  __syncwarp();
  f2 BX = 0ull, BY = 0ull, BZ = 0ull, TB = 0ull;
  npp += (t.valid && t.rep == 0) ? (unsigned)nsrc : 0u;
  const int np = (nsrc + 1) >> 1;
  if (any_near) {
#pragma unroll U
    for (int p = t.rep; p < np; p += t.nrep) pp_pair(a, t, S, p, BX, BY, BZ, TB, npp);
  } else {
#pragma unroll U
    for (int p = t.rep; p < np; p += t.nrep) pp_pair_far(t, S, p, BX, BY, BZ, TB);
  }
  __syncwarp();
  fold_pairs(t, BX, BY, BZ, TB);
}

// ---- particle-node batch (monopole + traceless quadrupole) ---------------
// a += -M r/r^3 + Q.r/r^5 - (5/2)(r.Q.r) r/r^7, r = x_i - com, for the two
// nodes of pair slot p (the stage holds -M)
__device__ __forceinline__ void node_pair(Target &t, const StageND32 &S, int p, f2 &BX,
                                          f2 &BY, f2 &BZ, f2 &TB) {
  const ulonglong2 hxy = S.hxy[p], hzw = S.hzw[p], lxy = S.lxy[p], lzw = S.lzw[p];
  const ulonglong2 q0xy = S.q0xy[p], q0zw = S.q0zw[p], q1xy = S.q1xy[p];
  const f2 dx = add2(sub2(t.X, hxy.x), sub2(t.XL, lxy.x));
  const f2 dy = add2(sub2(t.Y, hxy.y), sub2(t.YL, lxy.y));
  const f2 dz = add2(sub2(t.Z, hzw.x), sub2(t.ZL, lzw.x));
  const f2 r2 = fma2(dx, dx, fma2(dy, dy, mul2(dz, dz)));
  const f2 rinv = f2_pk(rsqrt_normal(fmaxf(f2_lo(r2), 1e-30f)),
                        rsqrt_normal(fmaxf(f2_hi(r2), 1e-30f)));
  const f2 rinv2 = mul2(rinv, rinv);
  const f2 rinv3 = mul2(rinv2, rinv);
  const f2 rinv5 = mul2(rinv3, rinv2);
  // q0xy = (xx, yy), q0zw = (zz, xy), q1xy = (xz, yz)
  const f2 qx = fma2(q0xy.x, dx, fma2(q0zw.y, dy, mul2(q1xy.x, dz)));
  const f2 qy = fma2(q0zw.y, dx, fma2(q0xy.y, dy, mul2(q1xy.y, dz)));
  const f2 qz = fma2(q1xy.x, dx, fma2(q1xy.y, dy, mul2(q0zw.x, dz)));
  const f2 rqr = fma2(dx, qx, fma2(dy, qy, mul2(dz, qz)));
  const f2 c = fma2(mul2(f2_dup(-2.5f), rqr), mul2(rinv5, rinv2), mul2(hzw.y, rinv3));
  BX = fma2(c, dx, fma2(qx, rinv5, BX));
  BY = fma2(c, dy, fma2(qy, rinv5, BY));
  BZ = fma2(c, dz, fma2(qz, rinv5, BZ));
  TB = fma2(hzw.y, rinv2, TB);  // -M / r^2
}

template <int U>
__device__ __forceinline__ void eval_nodes(const WalkArgs &a, Target &t,
                                           const int32_t *list, int nnd, void *stage,
                                           unsigned &npn) {
  StageND32 &S = *reinterpret_cast<StageND32 *>(stage);
  const int lane = threadIdx.x & 31;
  // lanes past the batch stage a massless, quadrupole-free dummy far away
  float4 hi = make_float4(1.0e18f, 1.0e18f, 1.0e18f, 0.f), lo = make_float4(0.f, 0.f, 0.f, 0.f);
  float4 q0 = lo, q1 = lo;
  if (lane < nnd) {
    const Mom32 *m = &a.mom32[list[lane]];
    hi = __ldg(&m->hi); lo = __ldg(&m->lo);
    q0 = __ldg(&m->q0); q1 = __ldg(&m->q1);
  }
  stage_put(S.hxy, lane, hi.x, hi.y);
  stage_put(S.hzw, lane, hi.z, -hi.w);
  stage_put(S.lxy, lane, lo.x, lo.y);
  stage_put(S.lzw, lane, lo.z, lo.w);
  stage_put(S.q0xy, lane, q0.x, q0.y);
  stage_put(S.q0zw, lane, q0.z, q0.w);
  stage_put(S.q1xy, lane, q1.x, q1.y);
  __syncwarp();
  f2 BX = 0ull, BY = 0ull, BZ = 0ull, TB = 0ull;
  npn += (t.valid && t.rep == 0) ? (unsigned)nnd : 0u;
  const int np = (nnd + 1) >> 1;
#pragma unroll U
  for (int p = t.rep; p < np; p += t.nrep) node_pair(t, S, p, BX, BY, BZ, TB);
  __syncwarp();
  // force sums as they are; the magnitude sum was of -M / r^2
  t.fold(f2_lo(BX) + f2_hi(BX), f2_lo(BY) + f2_hi(BY), f2_lo(BZ) + f2_hi(BZ));
  t.tabs -= f2_lo(TB) + f2_hi(TB);
}

// writes the target's acceleration; returns whether the target is to be
// redone in float-float
__device__ __forceinline__ bool write_result(const WalkArgs &a, Target &t) {
  if (!t.valid || t.rep != 0) return false;
  const double x = (double)t.ahx + (double)t.alx;
  const double y = (double)t.ahy + (double)t.aly;
  const double z = (double)t.ahz + (double)t.alz;
  const int32_t i = a.idx[t.self];
  a.ax[i] = a.G * x; a.ay[i] = a.G * y; a.az[i] = a.G * z;
  // FP32 terms carry ~1e-7 relative error each; where they cancel to a sum
  // much smaller than their magnitudes the target is redone in float-float
  const float amag = sqrtf((float)(x * x + y * y + z * z));
  return t.tabs > a.refine_cf * amag;
}

// ---- the traversal, shared by the group walk and the float-float redo ------
// Pops up to 32 nodes per round, decides opening on the integer grid, and
// hands full batches of 32 accepted nodes / leaf members to the evaluator.
// Returns false when the walk had to stop (capacity or round bound).
template <class Ev>
__device__ bool traverse(const WalkArgs &a, const GroupBox &gb, int32_t first, int32_t *stack,
                         int32_t *pp, int32_t *nd, int32_t *big,
                         const int64_t *s_bh, int64_t round_limit, Ev &ev) {
  const int lane = threadIdx.x & 31;
  const unsigned lt = (1u << lane) - 1u;
  int top = 1, npl = 0, nnd = 0, nbig = 0;
  int64_t rounds = 0;
  // sorted order keeps each segment contiguous, and segment d's root (level
  // 0, d-th in key order) is BFS node d: start at the root of the segment
  // that holds sorted particle `first`.  Every box inside the root cube lies
  // within 2^21 half cells of its centre on each axis, so when the root's
  // Barnes-Hut threshold exceeds 3 (2^21)^2 the root is opened for every
  // group: its children then start the stack, where the first round would
  // have pushed them
  const int32_t root = seg_at(a.seg, first);
  const int4 rc = __ldg(reinterpret_cast<const int4 *>(&a.node[root]) + 3);  // child0, nchild
  if (s_bh[0] > (3ll << 42) && rc.y > 0) {
    if (lane < rc.y) stack[lane] = rc.x + lane;
    top = rc.y;
  } else if (lane == 0) {
    stack[0] = root;
  }
  __syncwarp();
  while (top > 0) {
    if (++rounds > round_limit) {
      if (lane == 0) dev_fail(a.st, P3T_ERR_TIMEOUT, 43, 0);
      return false;
    }
    const int k = top < 32 ? top : 32;
    top -= k;
    int32_t id = -1;
    bool acc_node = false, open_leaf = false, open_inner = false;
    int32_t child0 = 0, nchild = 0, first = 0, count = 0;
    if (lane < k) {
      id = stack[top + lane];
      const int4 *r = reinterpret_cast<const int4 *>(&a.node[id]);
      const int4 q0 = __ldg(r), q1 = __ldg(r + 1), q2 = __ldg(r + 2), q3 = __ldg(r + 3);
      // (i) Barnes-Hut on the grid: half units, group cells [2 qlo, 2 qhi + 2]
      int64_t d2 = 0, g2 = 0;
      {
        int32_t d = max(0, max(2 * gb.qlo0 - q2.x, q2.x - (2 * gb.qhi0 + 2)));
        d2 += (int64_t)d * d;
        d = max(0, max(2 * gb.qlo1 - q2.y, q2.y - (2 * gb.qhi1 + 2)));
        d2 += (int64_t)d * d;
        d = max(0, max(2 * gb.qlo2 - q2.z, q2.z - (2 * gb.qhi2 + 2)));
        d2 += (int64_t)d * d;
      }
      // (ii) cut-off reach: lower-bound gap against the larger search reach
      {
        int32_t e = max(0, max(q0.x - gb.qhi0 - 2, gb.qlo0 - q1.x - 2));
        g2 += (int64_t)e * e;
        e = max(0, max(q0.y - gb.qhi1 - 2, gb.qlo1 - q1.y - 2));
        g2 += (int64_t)e * e;
        e = max(0, max(q0.z - gb.qhi2 - 2, gb.qlo2 - q1.z - 2));
        g2 += (int64_t)e * e;
      }
      const int64_t R = max(gb.R, q0.w);
      const bool open = (d2 < s_bh[q1.w]) || (g2 < R * R);
      child0 = q3.x; nchild = q3.y; first = q3.z; count = q3.w;
      acc_node = !open;
      open_leaf = open && nchild == 0;
      open_inner = open && nchild > 0;
    }
    // accepted nodes -> node list
    {
      const unsigned m = __ballot_sync(0xffffffffu, acc_node);
      if (acc_node) nd[nnd + __popc(m & lt)] = id;
      nnd += __popc(m);
    }
    // opened big leaves (> 32 members) -> their own list
    {
      const bool isbig = open_leaf && count > 32;
      const unsigned m = __ballot_sync(0xffffffffu, isbig);
      if (isbig) {
        const int slot = nbig + __popc(m & lt);
        if (slot < kBigCap) big[slot] = id;
      }
      nbig += __popc(m);
      if (isbig) open_leaf = false;
    }
    __syncwarp();  // every lane has read its stack entry before any push
    // children of opened inner nodes -> stack
    {
      int tot;
      const int c = open_inner ? nchild : 0;
      const int off = warp_excl_scan(c, &tot);
      if (top + tot > a.stack_cap) {
        if (lane == 0) dev_fail(a.st, P3T_ERR_CAPACITY, 40, top + tot);
        return false;
      }
      for (int q = 0; q < c; ++q) stack[top + off + q] = child0 + q;
      top += tot;
    }
    // members of opened leaves -> p-p list
    {
      int tot;
      const int c = open_leaf ? count : 0;
      const int off = warp_excl_scan(c, &tot);
      for (int q = 0; q < c; ++q) pp[npl + off + q] = first + q;
      npl += tot;
    }
    __syncwarp();
    if (nbig > kBigCap) {
      if (lane == 0) dev_fail(a.st, P3T_ERR_CAPACITY, 41, nbig);
      return false;
    }
    // evaluate full batches
    int o = 0;
    for (; nnd - o >= 32; o += 32) ev.nodes(nd + o, 32);
    if (o) {
      __syncwarp();
      const int rem = nnd - o;
      const int32_t v = lane < rem ? nd[o + lane] : 0;
      __syncwarp();
      if (lane < rem) nd[lane] = v;
      nnd = rem;
    }
    o = 0;
    for (; npl - o >= 32; o += 32) ev.pp(pp + o, 32);
    if (o) {
      __syncwarp();
      const int rem = npl - o;
      const int32_t v = lane < rem ? pp[o + lane] : 0;
      __syncwarp();
      if (lane < rem) pp[lane] = v;
      npl = rem;
    }
    __syncwarp();
  }
  if (nnd) ev.nodes(nd, nnd);
  if (npl) ev.pp(pp, npl);
  // big leaves, 32 members at a time, straight from their index range
  for (int b = 0; b < nbig; ++b) {
    const TreeNode &B = a.node[big[b]];
    for (int32_t s0 = B.first; s0 < B.first + B.count; s0 += 32) {
      const int ns = min(32, B.first + B.count - s0);
      __syncwarp();
      if (lane < ns) pp[lane] = s0 + lane;
      __syncwarp();
      ev.pp(pp, ns);
    }
  }
  __syncwarp();
  return true;
}

// up to 32 targets of a group (each on nrep lanes), batches staged in shared
// memory, U pair slots in flight
template <int U>
struct GroupEval {
  const WalkArgs &a;
  Target &t;
  void *stage;
  const FarBox &box;
  unsigned &npp, &npn;
  __device__ void nodes(const int32_t *list, int n) { eval_nodes<U>(a, t, list, n, stage, npn); }
  __device__ void pp(const int32_t *list, int n) {
    eval_pp<U>(a, t, list, n, stage, box, npp);
  }
};

// the walk's FarBox from its (valid) targets, written by lane 0
__device__ __forceinline__ void far_box(const Target &t, FarBox &b) {
  const float x = f2_lo(t.X) + f2_lo(t.XL), y = f2_lo(t.Y) + f2_lo(t.YL),
              z = f2_lo(t.Z) + f2_lo(t.ZL);
  const float inf = __int_as_float(0x7f800000);
  float lo0 = t.valid ? x : inf, lo1 = t.valid ? y : inf, lo2 = t.valid ? z : inf;
  float hi0 = t.valid ? x : -inf, hi1 = t.valid ? y : -inf, hi2 = t.valid ? z : -inf;
  const float ro = 1.0f / t.inv_ro;
  float R2 = t.valid ? fmaxf(t.rs2, ro * ro * 1.00001f) : 0.f;
  float am = t.valid ? fmaxf(fabsf(x), fmaxf(fabsf(y), fabsf(z))) : 0.f;
  for (int o = 16; o > 0; o >>= 1) {
    lo0 = fminf(lo0, __shfl_xor_sync(0xffffffffu, lo0, o));
    lo1 = fminf(lo1, __shfl_xor_sync(0xffffffffu, lo1, o));
    lo2 = fminf(lo2, __shfl_xor_sync(0xffffffffu, lo2, o));
    hi0 = fmaxf(hi0, __shfl_xor_sync(0xffffffffu, hi0, o));
    hi1 = fmaxf(hi1, __shfl_xor_sync(0xffffffffu, hi1, o));
    hi2 = fmaxf(hi2, __shfl_xor_sync(0xffffffffu, hi2, o));
    R2 = fmaxf(R2, __shfl_xor_sync(0xffffffffu, R2, o));
    am = fmaxf(am, __shfl_xor_sync(0xffffffffu, am, o));
  }
  __syncwarp();
  if ((threadIdx.x & 31) == 0) {
    b.lo[0] = lo0; b.lo[1] = lo1; b.lo[2] = lo2;
    b.hi[0] = hi0; b.hi[1] = hi1; b.hi[2] = hi2;
    b.R2 = R2;
    b.amax = am;
  }
  __syncwarp();
}

__device__ __forceinline__ FF ff_shfl(FF a, int src) {
  return {__shfl_sync(0xffffffffu, a.h, src), __shfl_sync(0xffffffffu, a.l, src)};
}

// one target, all 32 lanes, float-float (the refinement of ill-conditioned
// targets): relative coordinates, r^2, 1/r, masses, monopoles and the sums in
// float-float (terms to ~1e-13 of themselves); the changeover factor K and
// the quadrupole correction in FP32 (exact K = 1 beyond r_out)
struct RefineEval {
  const WalkArgs &a;
  float xh, yh, zh, xl, yl, zl, inv_ro;
  FF ax, ay, az;
  int s0, ds;  // this lane's entries of a batch: s0, s0 + ds, ...
  __device__ void term(FF dx, FF dy, FF dz, FF m, float k_inv_ro, bool pp, const float4 q0,
                       const float4 q1) {
    const FF r2 = ff_add(ff_add(ff_mul(dx, dx), ff_mul(dy, dy)), ff_mul(dz, dz));
    if (r2.h == 0.0f) return;  // the target itself
    const FF ri = ff_rsqrt(r2);
    const FF ri3 = ff_mul(ff_mul(ri, ri), ri);
    float K = 1.0f;
    if (pp) {
      const float y = r2.h * ri.h * k_inv_ro;
      const float x = __saturatef(fmaf(y, a.inv1mg_f, a.mgi_f));
      const float x2 = x * x;
      K = (x2 * x2) * fmaf(fmaf(fmaf(-20.f, x, 70.f), x, -84.f), x, 35.f);
      if (K == 0.0f) return;
    }
    const FF f = ff_mul(ff_mulf(m, K), ri3);  // m K / r^3
    ax = ff_add(ax, ff_mul(f, {-dx.h, -dx.l}));
    ay = ff_add(ay, ff_mul(f, {-dy.h, -dy.l}));
    az = ff_add(az, ff_mul(f, {-dz.h, -dz.l}));
    if (!pp) {  // Q.r / r^5 - (5/2) (r.Q.r) r / r^7 in FP32
      const float ddx = dx.h, ddy = dy.h, ddz = dz.h, rinv = ri.h;
      const float rinv2 = rinv * rinv, rinv5 = rinv2 * rinv2 * rinv;
      const float qx = fmaf(q0.x, ddx, fmaf(q0.w, ddy, q1.x * ddz));
      const float qy = fmaf(q0.w, ddx, fmaf(q0.y, ddy, q1.y * ddz));
      const float qz = fmaf(q1.x, ddx, fmaf(q1.y, ddy, q0.z * ddz));
      const float rqr = fmaf(ddx, qx, fmaf(ddy, qy, ddz * qz));
      const float c = -2.5f * rqr * rinv5 * rinv2;
      ax = ff_add(ax, ff_fast(fmaf(c, ddx, qx * rinv5), 0.0f));
      ay = ff_add(ay, ff_fast(fmaf(c, ddy, qy * rinv5), 0.0f));
      az = ff_add(az, ff_fast(fmaf(c, ddz, qz * rinv5), 0.0f));
    }
  }
  __device__ void pp(const int32_t *list, int n) {
    const float4 z4 = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int s = s0; s < n; s += ds) {
      const int32_t j = list[s];
      const float4 A = __ldg(&a.spA[j]), B = __ldg(&a.spB[j]);
      const FF dx = ff_add({xh, xl}, {-A.x, -B.x});
      const FF dy = ff_add({yh, yl}, {-A.y, -B.y});
      const FF dz = ff_add({zh, zl}, {-A.z, -B.z});
      term(dx, dy, dz, ff_fast(A.w, __ldg(&a.sml[j])), fminf(inv_ro, B.w), true, z4, z4);
    }
  }
  __device__ void nodes(const int32_t *list, int n) {
    for (int s = s0; s < n; s += ds) {
      const Mom32 *m = &a.mom32[list[s]];
      const float4 hi = __ldg(&m->hi), lo = __ldg(&m->lo);
      const FF dx = ff_add({xh, xl}, {-hi.x, -lo.x});
      const FF dy = ff_add({yh, yl}, {-hi.y, -lo.y});
      const FF dz = ff_add({zh, zl}, {-hi.z, -lo.z});
      term(dx, dy, dz, ff_fast(hi.w, lo.w), 0.0f, false, __ldg(&m->q0), __ldg(&m->q1));
    }
  }
};

// Float-float redo of the ill-conditioned targets of one walk (lanes with
// `redo` set), right after it: the same group box, hence the same interaction
// list, walked once for all of them.  With k such targets each takes
// floor(32 / k) lanes that split every batch (lane j + q k takes entries q,
// q + 32 / k, ... for target j); the lanes' float-float sums are added in
// replica order.
__device__ bool refine_group(const WalkArgs &a, const GroupBox &gb, bool redo, int32_t self,
                             int32_t first, int32_t *stack, int32_t *pp, int32_t *nd,
                             int32_t *big, const int64_t *s_bh, int64_t round_limit) {
  const int lane = threadIdx.x & 31;
  const unsigned todo = __ballot_sync(0xffffffffu, redo);
  const int k = __popc(todo);
  if (k == 0) return true;
  const int nrep = 32 / k, rep = lane / k, j = lane - rep * k;
  // lane of the j-th flagged target
  unsigned m = todo;
  for (int q = 0; q < j; ++q) m &= m - 1;
  const int32_t ti = __shfl_sync(0xffffffffu, self, __ffs(m) - 1);
  const bool valid = rep < nrep;
  const float4 A = a.spA[ti], B = a.spB[ti];
  RefineEval ev{a, A.x, A.y, A.z, B.x, B.y, B.z, B.w, {0.f, 0.f}, {0.f, 0.f}, {0.f, 0.f},
                valid ? rep : 32, nrep};
  if (!traverse(a, gb, first, stack, pp, nd, big, s_bh, round_limit, ev)) return false;
  // a target's own entry is skipped (r = 0)
  for (int q = 1; q < nrep; ++q) {
    const int src = lane < k ? lane + q * k : lane;
    const FF bx = ff_shfl(ev.ax, src), by = ff_shfl(ev.ay, src), bz = ff_shfl(ev.az, src);
    if (lane < k) {
      ev.ax = ff_add(ev.ax, bx);
      ev.ay = ff_add(ev.ay, by);
      ev.az = ff_add(ev.az, bz);
    }
  }
  if (lane < k) {
    const int32_t i = a.idx[ti];
    a.ax[i] = a.G * ((double)ev.ax.h + (double)ev.ax.l);
    a.ay[i] = a.G * ((double)ev.ay.h + (double)ev.ay.l);
    a.az[i] = a.G * ((double)ev.az.h + (double)ev.az.l);
  }
  return true;
}

// the warp's interaction counts to the caller's: a lane that met its target's
// own entry holds npp below zero, the warp sum is taken modulo 2^32, where a
// warp's true count fits
__device__ __forceinline__ void add_counts(const WalkArgs &a, unsigned p, unsigned q) {
  if (!a.counts) return;
  p = __reduce_add_sync(0xffffffffu, p);
  q = __reduce_add_sync(0xffffffffu, q);
  if ((threadIdx.x & 31) == 0) {
    atomicAdd(&a.counts[0], (unsigned long long)p);
    atomicAdd(&a.counts[1], (unsigned long long)q);
  }
}

// Two forms of the mixed walk, the same arithmetic in the same order.  Many
// units of work (U = 1): 80 registers, six blocks an SM, one pair slot at a
// time; a second slot in flight costs registers and is slower (N = 1e6: 1,219
// us, 1,514 with four blocks of two slots).  Fewer units than warps (U = 4): a
// unit has a sub-partition nearly to itself and its time is the latency of its
// own chain, which four slots in flight shorten.
constexpr int kFewU = 4, kManyBlocks = 6, kFewBlocks = 3;
template <int U>
__global__ void __launch_bounds__(kWarps * 32, U == 1 ? kManyBlocks : kFewBlocks)
    k_walk(const WalkArgs a) {
  pdl_wait();
  __shared__ int32_t s_pp[kWarps][kPPCap];
  __shared__ int32_t s_nd[kWarps][kNDCap];
  __shared__ int32_t s_big[kWarps][kBigCap];
  __shared__ __align__(16) unsigned char s_stage[kWarps][kStageBytes];
  __shared__ int64_t s_bh[P3T_BITS + 1];
  __shared__ FarBox s_box[kWarps];
  if (threadIdx.x <= P3T_BITS) s_bh[threadIdx.x] = a.bh[threadIdx.x];
  __syncthreads();

  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  int32_t *stack = a.stack + ((int64_t)blockIdx.x * kWarps + w) * a.stack_cap;
  const int64_t nleaf = *a.d_nleaf;
  const int64_t round_limit = *a.d_nnode + 2;  // a node is pushed at most once per walk
  const int64_t paired = max((int64_t)0, nleaf - (int64_t)gridDim.x * kWarps);
  unsigned npp = 0, npn = 0;

  for (;;) {
    // work unit u: the first 32 targets of a target group or the rest of it
    // (empty for a group of at most 32): units of at most 32 targets keep the
    // warps' finishing times close.  A group's rest follows its first 32, which
    // meet much the same nodes, but for the last groups, as many as there are
    // warps: all their first 32, then their rests, mostly small, so that the end
    // has small units.  Force, rests at once / all at the end / this, wide disk: N =
    // 2e5 307 / 321 / 286 us, 3e5 456 / 434 / 430, 6e5 729 / 756 / 710, 1e6 1,243 /
    // 1,218 / 1,202; ring 1e5 330 / 248 / 240
    int64_t u = 0;
    if (lane == 0) u = atomicAdd(reinterpret_cast<unsigned long long *>(a.cursor), 1ull);
    u = __shfl_sync(0xffffffffu, u, 0);
    const int64_t v = u - 2 * paired;
    const bool rest = v < 0 ? (u & 1) : v >= nleaf - paired;
    const int64_t g = v < 0 ? u >> 1 : (rest ? v - nleaf + 2 * paired : v + paired);
    if (g >= nleaf) break;
    if (*(volatile int32_t *)&a.st->code != 0) break;
    const TreeNode &G = a.node[a.leaf_list[g]];
    const int32_t gfirst = G.first, gcount = G.count;
    const int32_t t0 = rest ? gfirst + 32 : gfirst;
    const int32_t t1 = rest ? gfirst + gcount : min(gfirst + gcount, gfirst + 32);
    if (t0 >= t1) continue;
    GroupBox gb;
    gb.load(G);
    bool ok = true;
    for (int32_t tb = t0; tb < t1 && ok; tb += 32) {
      const int k = min(32, t1 - tb);
      const int nrep = 32 / k, rep = lane / k;
      Target t;
      t.load(a, tb + (lane - rep * k), rep < nrep, rep < nrep ? rep : 0, nrep);
      far_box(t, s_box[w]);
      GroupEval<U> ev{a, t, s_stage[w], s_box[w], npp, npn};
      ok = traverse(a, gb, gfirst, stack, s_pp[w], s_nd[w], s_big[w], s_bh, round_limit, ev);
      if (ok) {
        t.reduce(k);
        const bool redo = write_result(a, t);
        ok = refine_group(a, gb, redo, t.self, gfirst, stack, s_pp[w], s_nd[w], s_big[w], s_bh,
                          round_limit);
      }
    }
    if (!ok) break;
  }
  add_counts(a, npp, npn);
}

// ---- the FP64 walk ------------------------------------------------------------
// Bound by the FP64 pipe (a warp instruction per 19 cycles of an SM), with
// issue slots to spare.  A chunk of up to kChunk targets of a group is walked
// at a time; a batch of 32 list entries stands in the lanes' registers, one
// entry a lane, and the chunk's targets (in shared memory, read by broadcast)
// are taken in turn, each lane adding its entry's term to its own partial sum
// of that target in shared memory.  Every lane carries an entry whatever the
// group's size, and a target's sum is 32 partial sums (entry position modulo
// 32, in list order) added in one fixed tree: it does not depend on the
// chunk, so the host may choose it by the size of the system.  A batch whose
// entries are all beyond every target's cut-off reach (decided in FP32 with a
// margin) skips the changeover and the candidate test; the factor K = 1
// would leave the same bits.  16 FP64 instructions a far pair, 30 a near one,
// 37 a node, every lane in use (with rsqrt() and one lane a target 0.6-0.9 of
// them): N = 1e5 ring, theta 0.5, 4,790 -> 2,700 us a walk (93 % of the FP64 pipe's
// instruction rate); 3 to 5 blocks an SM and chunks of 4 or 8 within 2 %.
constexpr int kChunk = 8;
constexpr int kWalk64Blocks = 4;
struct Targets64 {
  double x[kChunk], y[kChunk], z[kChunk], iro[kChunk];
  int32_t rs2[kChunk];  // leading bits of r_search^2
  double acc[kChunk * 3][33];  // a row's 32 partial sums (33: columns in different banks)
};

// FP32 box of the chunk and its largest max(r_search, r_out)^2, as FarBox
__device__ __forceinline__ void far_box64(const WalkArgs &a, int32_t t0, int nt, FarBox &b) {
  const int lane = threadIdx.x & 31;
  const int32_t i = t0 + min(lane, nt - 1);
  const float x = lead_float(a.sx[i], 0), y = lead_float(a.sy[i], 0), z = lead_float(a.sz[i], 0);
  const float ro = lead_float(a.sro[i], 0), rs = lead_float(a.srs[i], 0);
  float lo0 = x, lo1 = y, lo2 = z, hi0 = x, hi1 = y, hi2 = z;
  float R = fmaxf(ro, rs), am = fmaxf(fabsf(x), fmaxf(fabsf(y), fabsf(z)));
#pragma unroll
  for (int o = kChunk / 2; o > 0; o >>= 1) {
    lo0 = fminf(lo0, __shfl_xor_sync(0xffffffffu, lo0, o));
    lo1 = fminf(lo1, __shfl_xor_sync(0xffffffffu, lo1, o));
    lo2 = fminf(lo2, __shfl_xor_sync(0xffffffffu, lo2, o));
    hi0 = fmaxf(hi0, __shfl_xor_sync(0xffffffffu, hi0, o));
    hi1 = fmaxf(hi1, __shfl_xor_sync(0xffffffffu, hi1, o));
    hi2 = fmaxf(hi2, __shfl_xor_sync(0xffffffffu, hi2, o));
    R = fmaxf(R, __shfl_xor_sync(0xffffffffu, R, o));
    am = fmaxf(am, __shfl_xor_sync(0xffffffffu, am, o));
  }
  __syncwarp();
  if (lane == 0) {
    b.lo[0] = lo0; b.lo[1] = lo1; b.lo[2] = lo2;
    b.hi[0] = hi0; b.hi[1] = hi1; b.hi[2] = hi2;
    b.R2 = R;
    b.amax = am;
  }
  __syncwarp();
}
// whether a source is beyond every target's max(r_search, r_out) and its own:
// the gap to the box less 2^-18 of the coordinates' scale (their truncation to
// 20 bits), against the reach widened by 1e-5.  A gap whose square leaves FP32's
// range is not decided here: it would pass against a reach whose square does
__device__ __forceinline__ bool far_from64(const FarBox &b, double X, double Y, double Z,
                                           double ro, double rs) {
  const float x = lead_float(X, 0), y = lead_float(Y, 0), z = lead_float(Z, 0);
  const float m = 3.814697265625e-6f *
                  (b.amax + fmaxf(fabsf(x), fmaxf(fabsf(y), fabsf(z))));
  const float gx = fmaxf(fmaxf(b.lo[0] - x, x - b.hi[0]) - m, 0.f);
  const float gy = fmaxf(fmaxf(b.lo[1] - y, y - b.hi[1]) - m, 0.f);
  const float gz = fmaxf(fmaxf(b.lo[2] - z, z - b.hi[2]) - m, 0.f);
  const float R = fmaxf(b.R2, fmaxf(lead_float(ro, 0), lead_float(rs, 0))) * 1.00001f;
  const float d2 = gx * gx + gy * gy + gz * gz;
  return d2 > 1e-30f && d2 < 3e38f && d2 >= R * R;
}

// m r^-3 from r^2 (zero for r = 0 and where r^2 is infinite): the seed's y, y^2
// and e = 1 - r^2 y^2 and the result (see rsqrt_seed)
struct Inv3 {
  double y, y2, e, f;
};
__device__ __forceinline__ Inv3 inv_cube(double r2, double m) {
  Inv3 v;
  const RsqrtSeed s = rsqrt_seed(r2);
  v.y = s.y;
  v.y2 = s.y2;
  v.e = s.e;
  const double t = v.y2 * (v.y * m);
  v.f = fma(t * v.e, fma(1.875, v.e, 1.5), t);
  return v;
}
// min of two positive numbers and clamp to [0, 1], on the bit patterns (an FP64
// comparison takes an FP64 instruction)
__device__ __forceinline__ double min_pos(double a, double b) {
  return __double_as_longlong(a) < __double_as_longlong(b) ? a : b;
}
__device__ __forceinline__ double clamp01(double x) {
  const long long b = __double_as_longlong(x), one = 0x3ff0000000000000LL;
  return __longlong_as_double(b < 0 ? 0 : (b > one ? one : b));
}
// whether a clamped x lies strictly between 0 and 1
__device__ __forceinline__ bool inside01(double x) {
  return (unsigned long long)(__double_as_longlong(x) - 1) < 0x3fefffffffffffffULL;
}
// 1 / r to full precision
__device__ __forceinline__ double inv_r(const Inv3 &v) {
  return fma(v.y * v.e, fma(0.375, v.e, 0.5), v.y);
}

struct Eval64 {
  const WalkArgs &a;
  Targets64 &t;
  const FarBox &box;
  int32_t t0;
  int nt;
  unsigned &npp, &npn;
  __device__ __forceinline__ void add(int i, double fx, double dx, double fy, double dy, double fz,
                                      double dz) {
    const int lane = threadIdx.x & 31;
    t.acc[3 * i][lane] = fma(fx, dx, t.acc[3 * i][lane]);
    t.acc[3 * i + 1][lane] = fma(fy, dy, t.acc[3 * i + 1][lane]);
    t.acc[3 * i + 2][lane] = fma(fz, dz, t.acc[3 * i + 2][lane]);
  }
  __device__ void pp(const int32_t *list, int n) {
    const int lane = threadIdx.x & 31;
    const bool on = lane < n;
    const int32_t j = list[on ? lane : 0];
    const double X = a.sx[j], Y = a.sy[j], Z = a.sz[j], ro = a.sro[j], rs = a.srs[j];
    const double m = on ? -a.sm[j] : 0.0;
    npp += on ? (unsigned)nt : 0u;
    if (!__any_sync(0xffffffffu, on && !far_from64(box, X, Y, Z, ro, rs))) {
#pragma unroll 1
      for (int i = 0; i < nt; ++i) {
        const double dx = t.x[i] - X, dy = t.y[i] - Y, dz = t.z[i] - Z;
        const double f = inv_cube(fma(dx, dx, fma(dy, dy, dz * dz)), m).f;
        add(i, f, dx, f, dy, f, dz);
      }
      return;
    }
    const double iro = 1.0 / ro;
    const int32_t rs2 = __double2hiint(rs * rs);
#pragma unroll 1
    for (int i = 0; i < nt; ++i) {
      const double dx = t.x[i] - X, dy = t.y[i] - Y, dz = t.z[i] - Z;
      const double r2 = fma(dx, dx, fma(dy, dy, dz * dz));
      const Inv3 v = inv_cube(r2, m);
      // y = r / max(r_out,i, r_out,j) as r min(1 / r_out)
      const double y = (r2 * inv_r(v)) * min_pos(t.iro[i], iro);
      const double x = clamp01((y - a.gamma) * a.inv1mg);
      const double x2 = x * x;
      const double K = (x2 * x2) * fma(fma(fma(-20.0, x, 70.0), x, -84.0), x, 35.0);
      const double f = v.f * K;
      add(i, f, dx, f, dy, f, dz);
      // r < max(r_search) by the leading 32 bits (a superset; the exact test
      // follows in the neighbour search)
      if (on && __double2hiint(r2) <= max(t.rs2[i], rs2)) {
        if (j != t0 + i) record_candidate(a, t0 + i, j);
        else --npp;  // the target itself is not a pair
      }
    }
  }
  // a += -M r/r^3 + Q.r/r^5 - (5/2)(r.Q.r) r/r^7, r = x_i - com
  __device__ void nodes(const int32_t *list, int n) {
    const int lane = threadIdx.x & 31;
    const bool on = lane < n;
    const Mom64 *g = &a.mom64[list[on ? lane : 0]];
    const double2 c0 = __ldg(reinterpret_cast<const double2 *>(g)),
                  c1 = __ldg(reinterpret_cast<const double2 *>(g) + 1),
                  q0 = __ldg(reinterpret_cast<const double2 *>(g) + 2),
                  q1 = __ldg(reinterpret_cast<const double2 *>(g) + 3),
                  q2 = __ldg(reinterpret_cast<const double2 *>(g) + 4);
    const double M = on ? c1.y : 0.0;
    const double qxx = on ? q0.x : 0.0, qyy = on ? q0.y : 0.0, qzz = on ? q1.x : 0.0,
                 qxy = on ? q1.y : 0.0, qxz = on ? q2.x : 0.0, qyz = on ? q2.y : 0.0;
    npn += on ? (unsigned)nt : 0u;
#pragma unroll 1
    for (int i = 0; i < nt; ++i) {
      const double dx = t.x[i] - c0.x, dy = t.y[i] - c0.y, dz = t.z[i] - c1.x;
      const double r2 = fma(dx, dx, fma(dy, dy, dz * dz));
      const Inv3 v = inv_cube(r2, 1.0);
      const double ri3 = v.f, y2 = v.y2;
      const double ri2 = fma(y2, fma(v.e, v.e, v.e), y2);  // y^2 / (1 - e)
      const double qx = fma(qxx, dx, fma(qxy, dy, qxz * dz));
      const double qy = fma(qxy, dx, fma(qyy, dy, qyz * dz));
      const double qz = fma(qxz, dx, fma(qyz, dy, qzz * dz));
      const double s = fma(dx, qx, fma(dy, qy, dz * qz)) * ri2;
      const double A = fma(-2.5, s * ri2, -M) * ri3, B = ri3 * ri2;
      add(i, A, dx, A, dy, A, dz);
      add(i, B, qx, B, qy, B, qz);
    }
  }
};

// the chunk's sums: the 32 partial sums of each row in one fixed tree (k +
// (k + 16), then 8, 4, 2, 1), a row a lane
__device__ __forceinline__ double row_sum(double *r) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1)
    for (int k = 0; k < o; ++k) r[k] += r[k + o];
  return r[0];
}

__global__ void __launch_bounds__(kWarps * 32) k_walk64(const WalkArgs a, int ct) {
  pdl_wait();
  __shared__ int32_t s_pp[kWarps][kPPCap];
  __shared__ int32_t s_nd[kWarps][kNDCap];
  __shared__ int32_t s_big[kWarps][kBigCap];
  __shared__ Targets64 s_t[kWarps];
  __shared__ int64_t s_bh[P3T_BITS + 1];
  __shared__ FarBox s_box[kWarps];
  if (threadIdx.x <= P3T_BITS) s_bh[threadIdx.x] = a.bh[threadIdx.x];
  __syncthreads();

  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  int32_t *stack = a.stack + ((int64_t)blockIdx.x * kWarps + w) * a.stack_cap;
  const int64_t ngroup = *a.d_nleaf;
  const int64_t round_limit = *a.d_nnode + 2;  // a node is pushed at most once per walk
  const int parts = (a.group_max + ct - 1) / ct;
  Targets64 &t = s_t[w];
  unsigned npp = 0, npn = 0;

  for (;;) {
    // work unit u: chunk u mod parts of target group u / parts (empty for the
    // smaller groups); the last chunk takes what an oversized leaf has left
    int64_t u = 0;
    if (lane == 0) u = atomicAdd(reinterpret_cast<unsigned long long *>(a.cursor), 1ull);
    u = __shfl_sync(0xffffffffu, u, 0);
    const int64_t g = u / parts;
    const int part = (int)(u - g * parts);
    if (g >= ngroup) break;
    if (*(volatile int32_t *)&a.st->code != 0) break;
    const TreeNode &G = a.node[a.leaf_list[g]];
    const int32_t gfirst = G.first, gend = G.first + G.count;
    const int32_t u0 = gfirst + part * ct;
    const int32_t u1 = part == parts - 1 ? gend : min(gend, u0 + ct);
    if (u0 >= u1) continue;
    GroupBox gb;
    gb.load(G);
    bool ok = true;
    for (int32_t t0 = u0; t0 < u1 && ok; t0 += ct) {
      const int nt = min(ct, u1 - t0);
      if (lane < nt) {
        const int32_t i = t0 + lane;
        t.x[lane] = a.sx[i]; t.y[lane] = a.sy[i]; t.z[lane] = a.sz[i];
        t.iro[lane] = 1.0 / a.sro[i];
        t.rs2[lane] = __double2hiint(a.srs[i] * a.srs[i]);
      }
      for (int k = 0; k < 3 * nt; ++k) t.acc[k][lane] = 0.0;
      far_box64(a, t0, nt, s_box[w]);
      Eval64 ev{a, t, s_box[w], t0, nt, npp, npn};
      ok = traverse(a, gb, gfirst, stack, s_pp[w], s_nd[w], s_big[w], s_bh, round_limit, ev);
      __syncwarp();
      if (ok)
        for (int k = lane; k < 3 * nt; k += 32) {
          const int i = k / 3, c = k - 3 * i;
          (c == 0 ? a.ax : (c == 1 ? a.ay : a.az))[a.idx[t0 + i]] = a.G * row_sum(t.acc[k]);
        }
      __syncwarp();
    }
    if (!ok) break;
  }
  add_counts(a, npp, npn);
}

// ---- adjoint of the tree walk (FP64 path) -----------------------------------
// The vector-Jacobian product of the soft force of Eq. softforce as the tree
// gives it, with the tree and the interaction lists held fixed: a second walk
// of the same tree from the same group boxes meets the same lists.  With
// L = sum_i lam_i . a_i (lam_i = s times the caller's velocity adjoint):
//   p-p term a_i += -G m_j K(y) r / r^3, r = x_i - x_j, y = r / r_out,ij:
//     dL/dx_i += J lam_i, dL/dx_j -= J lam_i, dL/dm_j += lam_i . (-G K r / r^3),
//     J = -G m_j (phi I + psi r r^T), phi = K / r^3,
//     psi = K'(y) / (r_out,ij r^4) - 3 K / r^5;
//   node term a_i += G [-M r / r^3 + Q r / r^5 - (5/2) (r.Q.r) r / r^7],
//     r = x_i - c: dL/dx_i += g, dL/dc -= g, with g = grad_r (lam_i . a),
//     and dL/dM, dL/dQ accumulated per node;
// the node adjoints then reach the member particles through M = sum m_k,
// c = sum m_k x_k / M, Q = sum m_k (3 d d^T - d^2 I), d = x_k - c (the
// derivative of Q through c vanishes, as sum m_k d_k = 0).  The layout of the
// FP64 walk: a lane per source or node, the targets of a chunk in turn, so
// that what the chunk's targets add to a source or node is summed in that
// lane's registers and goes to the global sums in one FP64 atomic per value
// and chunk (their order follows the walks' order, so the last bits can
// differ from run to run), and what the lanes add to a target in shared
// memory.  With lam' = G lam (lam scaled), z = r.Q.r / r^2, the node's
//   g = r^-5 [Q lam' + cl lam' + cr r + cq Q r], cl = -M r^2 - 5/2 z,
//   cr = 3 M lam'.r + (35/2 z lam'.r - 5 lam'.Q r) / r^2, cq = -5 lam'.r / r^2,
//   dL/dQ_ab = r^-5 sym(k_a r_b), k = lam' + cq/2 r:
// 84 FP64 instructions a node term and 33 a far pair (N = 10,000: 6,240 -> 600
// us a call), where one lane a target
// with a warp reduction per source took about 180 and 60 at half the lanes.
struct VjpOut {
  const double *lx, *ly, *lz;  // velocity adjoints, caller order
  double s;                    // scale (the kick's time step)
  double *gx, *gy, *gz, *gm;   // accumulated position and mass adjoints, caller order
  double *nadj;                // per node: dL/dc (3), dL/dM, dL/dQ (xx yy zz xy xz yz)
};

struct TargetsVjp {
  double x[kChunk], y[kChunk], z[kChunk], iro[kChunk];
  double lx[kChunk], ly[kChunk], lz[kChunk];  // s G lam
  double acc[kChunk * 3][33];
};

struct VjpEval {
  const WalkArgs &a;
  const VjpOut &o;
  TargetsVjp &t;
  const FarBox &box;
  int32_t t0;
  int nt;
  __device__ __forceinline__ void add(int i, double f, double vx, double vy, double vz) {
    const int lane = threadIdx.x & 31;
    t.acc[3 * i][lane] = fma(f, vx, t.acc[3 * i][lane]);
    t.acc[3 * i + 1][lane] = fma(f, vy, t.acc[3 * i + 1][lane]);
    t.acc[3 * i + 2][lane] = fma(f, vz, t.acc[3 * i + 2][lane]);
  }
  __device__ void nodes(const int32_t *list, int n) {
    const int lane = threadIdx.x & 31;
    const bool on = lane < n;
    const int32_t id = list[on ? lane : 0];
    const double2 *g = reinterpret_cast<const double2 *>(&a.mom64[id]);
    const double2 c0 = __ldg(g), c1 = __ldg(g + 1), q0 = __ldg(g + 2), q1 = __ldg(g + 3),
                  q2 = __ldg(g + 4);
    const double M = c1.y;
    double nx = 0.0, ny = 0.0, nz = 0.0, nM = 0.0;
    double nQ[6] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
#pragma unroll 1
    for (int i = 0; i < nt; ++i) {
      const double rx = t.x[i] - c0.x, ry = t.y[i] - c0.y, rz = t.z[i] - c1.x;
      const double lx = t.lx[i], ly = t.ly[i], lz = t.lz[i];
      const double r2 = fma(rx, rx, fma(ry, ry, rz * rz));
      const Inv3 v = inv_cube(r2, 1.0);
      const double ri3 = v.f, y2 = v.y2;
      const double ri2 = fma(y2, fma(v.e, v.e, v.e), y2);
      const double ri5 = ri3 * ri2;
      const double qx = fma(q0.x, rx, fma(q1.y, ry, q2.x * rz));
      const double qy = fma(q1.y, rx, fma(q0.y, ry, q2.y * rz));
      const double qz = fma(q2.x, rx, fma(q2.y, ry, q1.x * rz));
      const double z = fma(rx, qx, fma(ry, qy, rz * qz)) * ri2;
      const double lr = fma(lx, rx, fma(ly, ry, lz * rz));
      const double lq = fma(lx, qx, fma(ly, qy, lz * qz));
      const double l2 = lr * ri2;
      const double cl = fma(-2.5, z, -M * r2);
      const double cr = fma(ri2, fma(17.5 * z, lr, -5.0 * lq), 3.0 * M * lr);
      const double cq = -5.0 * l2, k5 = -2.5 * l2;
      const double hx = fma(cl, lx, fma(cr, rx, fma(cq, qx, fma(q0.x, lx, fma(q1.y, ly, q2.x * lz)))));
      const double hy = fma(cl, ly, fma(cr, ry, fma(cq, qy, fma(q1.y, lx, fma(q0.y, ly, q2.y * lz)))));
      const double hz = fma(cl, lz, fma(cr, rz, fma(cq, qz, fma(q2.x, lx, fma(q2.y, ly, q1.x * lz)))));
      // lanes past the batch repeat entry 0: their terms must not reach the target
      add(i, on ? ri5 : 0.0, hx, hy, hz);
      nx = fma(ri5, hx, nx); ny = fma(ri5, hy, ny); nz = fma(ri5, hz, nz);
      nM = fma(-lr, ri3, nM);
      const double kx = fma(k5, rx, lx), ky = fma(k5, ry, ly), kz = fma(k5, rz, lz);
      const double sx = ri5 * rx, sy = ri5 * ry, sz = ri5 * rz;
      nQ[0] = fma(kx, sx, nQ[0]); nQ[1] = fma(ky, sy, nQ[1]); nQ[2] = fma(kz, sz, nQ[2]);
      nQ[3] = fma(kx, sy, fma(ky, sx, nQ[3]));
      nQ[4] = fma(kx, sz, fma(kz, sx, nQ[4]));
      nQ[5] = fma(ky, sz, fma(kz, sy, nQ[5]));
    }
    if (on) {
      double *A = o.nadj + 10 * (int64_t)id;
      atomicAdd(&A[0], -nx); atomicAdd(&A[1], -ny); atomicAdd(&A[2], -nz); atomicAdd(&A[3], nM);
#pragma unroll
      for (int k = 0; k < 6; ++k) atomicAdd(&A[4 + k], nQ[k]);
    }
  }
  __device__ void pp(const int32_t *list, int n) {
    const int lane = threadIdx.x & 31;
    const bool on = lane < n;
    const int32_t j = list[on ? lane : 0];
    const double X = a.sx[j], Y = a.sy[j], Z = a.sz[j], ro = a.sro[j];
    const double m = on ? -a.sm[j] : 0.0;
    const bool near =
        __any_sync(0xffffffffu, on && !far_from64(box, X, Y, Z, ro, 0.0));
    const double iro = near ? 1.0 / ro : 0.0;
    // sum over the targets of K r^-3 lam' + psi (lam'.r) r, and of K r^-3 lam'.r
    double bx = 0.0, by = 0.0, bz = 0.0, bm = 0.0;
#pragma unroll 1
    for (int i = 0; i < nt; ++i) {
      const double rx = t.x[i] - X, ry = t.y[i] - Y, rz = t.z[i] - Z;
      const double lx = t.lx[i], ly = t.ly[i], lz = t.lz[i];
      const double r2 = fma(rx, rx, fma(ry, ry, rz * rz));
      const Inv3 v = inv_cube(r2, 1.0);
      const double y2 = v.y2;
      const double ri2 = fma(y2, fma(v.e, v.e, v.e), y2);
      double phi = v.f, psi;
      if (near) {
        // the target itself (r = 0) has phi = 0, and K' = 0 at both ends also
        // where 1 / r_out is infinite
        const double irot = min_pos(t.iro[i], iro);
        const double yv = (r2 * inv_r(v)) * irot;
        const double x = clamp01((yv - a.gamma) * a.inv1mg);
        const double x2 = x * x, u = 1.0 - x;
        const double K = (x2 * x2) * fma(fma(fma(-20.0, x, 70.0), x, -84.0), x, 35.0);
        const double dK = (140.0 * a.inv1mg) * ((x2 * x) * (u * u * u)) * (inside01(x) ? irot : 0.0);
        psi = fma(dK, ri2 * ri2, -3.0 * K * (phi * ri2));
        phi *= K;
        if (__double_as_longlong(x) == 0) phi = psi = 0.0;  // also where r^-3 is infinite
      } else {
        psi = -3.0 * (phi * ri2);
      }
      const double lr = fma(lx, rx, fma(ly, ry, lz * rz));
      const double pl = psi * lr;
      const double tx = fma(pl, rx, phi * lx), ty = fma(pl, ry, phi * ly), tz = fma(pl, rz, phi * lz);
      add(i, m, tx, ty, tz);
      bx += tx; by += ty; bz += tz;
      bm = fma(-phi, lr, bm);
    }
    if (on) {
      const int32_t i = a.idx[j];
      atomicAdd(&o.gx[i], -m * bx); atomicAdd(&o.gy[i], -m * by); atomicAdd(&o.gz[i], -m * bz);
      atomicAdd(&o.gm[i], bm);
    }
  }
};

__global__ void __launch_bounds__(kWarps * 32) k_walk_vjp(const WalkArgs a, int ct, const VjpOut o) {
  pdl_wait();
  __shared__ int32_t s_pp[kWarps][kPPCap];
  __shared__ int32_t s_nd[kWarps][kNDCap];
  __shared__ int32_t s_big[kWarps][kBigCap];
  __shared__ TargetsVjp s_t[kWarps];
  __shared__ int64_t s_bh[P3T_BITS + 1];
  __shared__ FarBox s_box[kWarps];
  if (threadIdx.x <= P3T_BITS) s_bh[threadIdx.x] = a.bh[threadIdx.x];
  __syncthreads();
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  int32_t *stack = a.stack + ((int64_t)blockIdx.x * kWarps + w) * a.stack_cap;
  const int64_t ngroup = *a.d_nleaf;
  const int64_t round_limit = *a.d_nnode + 2;
  const int parts = (a.group_max + ct - 1) / ct;  // as k_walk64
  TargetsVjp &t = s_t[w];
  for (;;) {
    int64_t u = 0;
    if (lane == 0) u = atomicAdd(reinterpret_cast<unsigned long long *>(a.cursor), 1ull);
    u = __shfl_sync(0xffffffffu, u, 0);
    const int64_t g = u / parts;
    const int part = (int)(u - g * parts);
    if (g >= ngroup) break;
    if (*(volatile int32_t *)&a.st->code != 0) break;
    const TreeNode &G = a.node[a.leaf_list[g]];
    const int32_t gfirst = G.first, gend = G.first + G.count;
    const int32_t u0 = gfirst + part * ct;
    const int32_t u1 = part == parts - 1 ? gend : min(gend, u0 + ct);
    if (u0 >= u1) continue;
    GroupBox gb;
    gb.load(G);
    bool ok = true;
    for (int32_t t0 = u0; t0 < u1 && ok; t0 += ct) {
      const int nt = min(ct, u1 - t0);
      if (lane < nt) {
        const int32_t k = t0 + lane, i = a.idx[k];
        t.x[lane] = a.sx[k]; t.y[lane] = a.sy[k]; t.z[lane] = a.sz[k];
        t.iro[lane] = 1.0 / a.sro[k];
        const double sg = o.s * a.G;
        t.lx[lane] = sg * o.lx[i]; t.ly[lane] = sg * o.ly[i]; t.lz[lane] = sg * o.lz[i];
      }
      for (int k = 0; k < 3 * nt; ++k) t.acc[k][lane] = 0.0;
      far_box64(a, t0, nt, s_box[w]);
      VjpEval ev{a, o, t, s_box[w], t0, nt};
      ok = traverse(a, gb, gfirst, stack, s_pp[w], s_nd[w], s_big[w], s_bh, round_limit, ev);
      __syncwarp();
      if (ok)
        for (int k = lane; k < 3 * nt; k += 32) {
          const int i = k / 3, c = k - 3 * i;
          atomicAdd(&(c == 0 ? o.gx : (c == 1 ? o.gy : o.gz))[a.idx[t0 + i]], row_sum(t.acc[k]));
        }
      __syncwarp();
    }
    if (!ok) break;
  }
}

// Node adjoints to the member particles.  With g = A_com / M and T the symmetric
// matrix of the quadrupole's part (T_xx = 6 A_xx - 2 tr A, T_xy = 3 A_xy, ...) a
// node adds, at d = x_k - com, A_M + g.d + d.T.d / 2 to dL/dm_k and m_k (g + T d)
// to dL/dx_k.  Every member of a leaf has the same ancestors, so a warp takes a
// leaf: each lane moves one ancestor's polynomial to the leaf's first member,
// ten lanes add the ten coefficients, leaf to root, and each lane evaluates
// the sum at a member.  Some 90 FP64 instructions a leaf, 75 a member's
// ancestor when every member climbed for itself.  Measured, N = 1e4: 119
// -> 18.5 us.
constexpr int kAncestors = 32;  // at least P3T_BITS + 1
__global__ void __launch_bounds__(128)
k_node_adjoint(const int64_t *d_nleaf, const int32_t *leaf_list, const TreeNode *node,
               const Mom64 *mom, const double *nadj, const double *sx, const double *sy,
               const double *sz, const double *sm, const int32_t *idx, double *gx, double *gy,
               double *gz, double *gm) {
  pdl_wait();
  __shared__ double s_v[4][10][kAncestors], s_c[4][10];
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  double (*v)[kAncestors] = s_v[w];
  const int64_t nleaf = *d_nleaf, nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t b = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5; b < nleaf; b += nwarps) {
    const int32_t leaf = leaf_list[b], first = node[leaf].first, count = node[leaf].count;
    int depth = 0;
    int32_t mine = -1;
    for (int32_t n = leaf; n >= 0 && depth < kAncestors; n = node[n].parent, ++depth)
      if (lane == depth) mine = n;
    const double rx = sx[first], ry = sy[first], rz = sz[first];
    if (mine >= 0) {
      const double *A = nadj + 10 * (int64_t)mine;
      const Mom64 &M = mom[mine];
      const double iM = 1.0 / M.M, dx = rx - M.cx, dy = ry - M.cy, dz = rz - M.cz;
      const double tr2 = 2.0 * (A[4] + A[5] + A[6]);
      const double xx = fma(6.0, A[4], -tr2), yy = fma(6.0, A[5], -tr2),
                   zz = fma(6.0, A[6], -tr2), xy = 3.0 * A[7], xz = 3.0 * A[8], yz = 3.0 * A[9];
      const double tx = fma(xx, dx, fma(xy, dy, xz * dz)), ty = fma(xy, dx, fma(yy, dy, yz * dz)),
                   tz = fma(xz, dx, fma(yz, dy, zz * dz));
      const double px = A[0] * iM, py = A[1] * iM, pz = A[2] * iM;
      v[0][lane] = A[3] + fma(fma(0.5, tx, px), dx, fma(fma(0.5, ty, py), dy, fma(0.5, tz, pz) * dz));
      v[1][lane] = px + tx; v[2][lane] = py + ty; v[3][lane] = pz + tz;
      v[4][lane] = xx; v[5][lane] = yy; v[6][lane] = zz;
      v[7][lane] = xy; v[8][lane] = xz; v[9][lane] = yz;
    }
    __syncwarp();
    if (lane < 10) {
      double c = v[lane][0];
      for (int q = 1; q < depth; ++q) c += v[lane][q];
      s_c[w][lane] = c;
    }
    __syncwarp();
    const double *c = s_c[w];
    for (int32_t k = first + lane; k < first + count; k += 32) {
      const double dx = sx[k] - rx, dy = sy[k] - ry, dz = sz[k] - rz, mk = sm[k];
      const double tx = fma(c[4], dx, fma(c[7], dy, c[8] * dz)),
                   ty = fma(c[7], dx, fma(c[5], dy, c[9] * dz)),
                   tz = fma(c[8], dx, fma(c[9], dy, c[6] * dz));
      const int32_t i = idx[k];
      gx[i] = fma(mk, c[1] + tx, gx[i]);
      gy[i] = fma(mk, c[2] + ty, gy[i]);
      gz[i] = fma(mk, c[3] + tz, gz[i]);
      gm[i] += c[0] + fma(fma(0.5, tx, c[1]), dx,
                          fma(fma(0.5, ty, c[2]), dy, fma(0.5, tz, c[3]) * dz));
    }
    __syncwarp();
  }
}

// after a walk: the candidates found to the device status (for growth on the
// host) and clamped for the neighbour search, the interaction counts to the
// caller's, and the walk's counters back to zero for the next one
// (cnt: [8] candidates, [9] clamped, [12] cursor, [25] p-p, [26] p-node)
__global__ void k_walk_post(int64_t *cnt, int64_t cand_cap, unsigned long long *counts,
                            DevStatus *st) {
  pdl_wait();
  const int64_t nc = cnt[8];
  st->cand_need = nc;
  if (nc > cand_cap) dev_fail(st, P3T_ERR_CAPACITY, 42, nc);
  cnt[9] = nc < cand_cap ? nc : cand_cap;
  if (counts) {
    counts[0] = (unsigned long long)cnt[25];
    counts[1] = (unsigned long long)cnt[26];
  }
  cnt[8] = cnt[12] = cnt[25] = cnt[26] = 0;
}

// T M^2 >= 2^K for T < 2^49, M < 2^53, K >= 0: the product formed exactly in
// three 64-bit limbs and compared with the power of two
bool prod_sq_ge_pow2(uint64_t T, uint64_t M, int K) {
  const unsigned __int128 a = (unsigned __int128)T * M;  // < 2^102
  const unsigned __int128 p0 = (unsigned __int128)(uint64_t)a * M;
  const unsigned __int128 p1 = (unsigned __int128)(uint64_t)(a >> 64) * M;
  const unsigned __int128 mid = (p0 >> 64) + (unsigned __int128)(uint64_t)p1;
  const uint64_t w[3] = {(uint64_t)p0, (uint64_t)mid,
                         (uint64_t)(p1 >> 64) + (uint64_t)(mid >> 64)};
  if (K >= 192) return false;
  for (int q = 2; q > K / 64; --q)
    if (w[q]) return true;
  return (w[K / 64] >> (K % 64)) != 0;
}

// Barnes-Hut threshold of a level: the smallest integer T with T theta^2 >=
// side^2, side = 2^(22 - l) half cells, so that the integer test d^2 < T is
// exactly side^2 > theta^2 d^2.  theta = M 2^E with M odd, so the condition
// is T M^2 >= 2^K, K = 2 (22 - l) - 2E.  The FP64 quotient side^2 / theta^2
// gives T to within one, and the exact product settles it.  Thresholds
// beyond 2^47 (above every squared distance on the grid, < 3 * 2^44) are
// clamped to 2^47; theta = 0 opens every node.
int64_t bh_threshold(double theta, int level) {
  const int64_t cap = (int64_t)1 << 47;
  if (!(theta > 0.0)) return cap;
  int e;
  uint64_t M = (uint64_t)ldexp(frexp(theta, &e), 53);
  int E = e - 53;
  while (!(M & 1u)) { M >>= 1; ++E; }
  const int K = 2 * (P3T_BITS + 1 - level) - 2 * E;
  if (K < 0) return 1;
  const double X = ldexp(1.0, 2 * (P3T_BITS + 1 - level)) / (theta * theta);
  if (X > (double)cap + 4.0) return cap;
  uint64_t T = (uint64_t)ceil(X);
  if (T < 1) T = 1;
  while (T > 1 && prod_sq_ge_pow2(T - 1, M, K)) --T;
  while (!prod_sq_ge_pow2(T, M, K)) ++T;
  return (int64_t)T < cap ? (int64_t)T : cap;
}

}  // namespace

// blocks of 4 warps resident per SM: the mixed walk is compiled for 6 (80
// registers; 30.5 KB of shared memory a block)
int p3t_walk_blocks_per_sm() { return kManyBlocks; }

// the walk's arguments for the tree of context c built from particles p
static WalkArgs walk_args(p3t_ctx *c, const p3t_particles *p) {
  WalkArgs a;
  a.node = c->node; a.mom64 = c->mom64; a.mom32 = c->mom32;
  a.leaf_list = c->group_list; a.d_nleaf = &c->counters[15]; a.d_nnode = &c->counters[3];
  a.sx = c->sx; a.sy = c->sy; a.sz = c->sz; a.sm = c->sm; a.sro = c->sro; a.srs = c->srs;
  a.spA = c->spA; a.spB = c->spB; a.srs32 = c->srs32; a.sml = c->sml;
  a.idx = c->idx;
  a.ax = a.ay = a.az = nullptr;
  a.stack = c->walk_stack; a.stack_cap = c->stack_cap;
  a.cand_i = c->cand_i; a.cand_j = c->cand_j; a.cand_cap = c->cand_cap;
  a.cand_count = reinterpret_cast<unsigned long long *>(&c->counters[8]);
  a.counts = nullptr;
  a.cursor = &c->counters[12];
  a.st = c->status;
  a.seg = SegView{c->seg_off, (int)c->nseg, p->n};
  a.group_max = c->prm.group_size > c->prm.leaf_size ? c->prm.group_size : c->prm.leaf_size;
  a.refine_cf = 32.0f;
  a.G = c->prm.G;
  a.gamma = c->prm.gamma;
  a.inv1mg = 1.0 / (1.0 - c->prm.gamma);
  a.inv1mg_f = (float)(1.0 / (1.0 - c->prm.gamma));
  a.mgi_f = (float)(-c->prm.gamma / (1.0 - c->prm.gamma));
  for (int l = 0; l <= P3T_BITS; ++l) a.bh[l] = bh_threshold(c->prm.theta, l);
  return a;
}

// particles an SM up to which the mixed walk takes its few-units form (about
// one unit a warp at three blocks an SM).  Force, few / many, wide disk: N =
// 3,001 96 / 107 us, 1e4 99 / 122, 3e4 116 / 133, 4.5e4 132 / 147, 6e4 194 / 184;
// ring: 3e4 117 / 138, 6e4 216 / 174, 1e5 439 / 247
constexpr int kFewTargets = 200;

// The FP64 walks' chunk of targets: up to kChunk at a time (one traversal
// serves them all, and in the VJP one set of atomics a node), fewer while a
// warp would get less than two chunks, so that small systems fill the card (N =
// 1,000: chunks of one target; from about 50,000 particles on the largest).
// Force / VJP with at least two, four and one chunk a warp: N = 1e4 216 / 461,
// 229 / 522, 223 / 435 us; 3e4 724 / 1,573, 716 / 1,593, 794 / 1,611
static int walk64_chunk(const p3t_ctx *c, unsigned blocks) {
  int ct = kChunk;
  while (ct > 1 && c->last_n < (int64_t)2 * ct * blocks * kWarps) ct >>= 1;
  return ct;
}
// their blocks per SM: kWalk64Blocks (12 warps hold the FP64 pipe busy through
// each other's traversals)
static unsigned walk64_blocks(const p3t_ctx *c, unsigned blocks) {
  const unsigned most = (unsigned)c->num_sms * kWalk64Blocks;
  return blocks < most ? blocks : most;
}

int p3t_run_soft_force_vjp_tree(p3t_ctx *c, const p3t_particles *p, double s,
                                const double *lx, const double *ly, const double *lz,
                                double *gx, double *gy, double *gz, double *gm,
                                cudaStream_t st) {
  WalkArgs a = walk_args(c, p);
  VjpOut o{lx, ly, lz, s, gx, gy, gz, gm, c->nadj};
  a.cursor = &c->counters[27];  // the forward walk leaves its own at zero
  P3T_CUDA_TRY(cudaMemsetAsync(c->nadj, 0, sizeof(double) * 10 * c->node_cap, st));
  P3T_CUDA_TRY(cudaMemsetAsync(a.cursor, 0, sizeof(int64_t), st));
  const unsigned blocks = walk64_blocks(c, (unsigned)(c->walk_warps / kWarps));
  pdl_launch(k_walk_vjp, dim3(blocks), dim3(kWarps * 32), 0, st, a, walk64_chunk(c, blocks), o);
  pdl_launch(k_node_adjoint, dim3((unsigned)(c->num_sms * 8)), dim3(128), 0, st, 
      &c->counters[2], c->leaf_list, c->node, c->mom64, c->nadj, c->sx, c->sy, c->sz, c->sm,
      c->idx, gx, gy, gz, gm);
  p3t_note_launches(3);
  return cudaGetLastError() == cudaSuccess ? P3T_OK : P3T_ERR_CUDA;
}

int p3t_run_soft_force(p3t_ctx *c, const p3t_particles *p, double *ax,
                       double *ay, double *az, uint64_t *counts,
                       cudaStream_t s) {
  WalkArgs a = walk_args(c, p);
  a.ax = ax; a.ay = ay; a.az = az;
  a.counts = reinterpret_cast<unsigned long long *>(&c->counters[25]);
  unsigned blocks = (unsigned)(c->walk_warps / kWarps);
  if (c->walk_bps > 0 && (int64_t)c->num_sms * c->walk_bps < (int64_t)blocks)
    blocks = (unsigned)(c->num_sms * c->walk_bps);
  if (c->prm.precision == P3T_MIXED) {
    // one target per lane (or several lanes per target): two targets per
    // lane (a 64-target group walked once) was measured slower than two
    // walks of 32 (register pressure, longer chains)
    if (c->last_n <= (int64_t)kFewTargets * c->num_sms) {
      blocks = std::min(blocks, (unsigned)(c->num_sms * kFewBlocks));
      pdl_launch(k_walk<kFewU>, dim3(blocks), dim3(kWarps * 32), 0, s, a);
    } else {
      pdl_launch(k_walk<1>, dim3(blocks), dim3(kWarps * 32), 0, s, a);
    }
  } else {
    blocks = walk64_blocks(c, blocks);
    pdl_launch(k_walk64, dim3(blocks), dim3(kWarps * 32), 0, s, a, walk64_chunk(c, blocks));
  }
  pdl_launch(k_walk_post, dim3(1), dim3(1), 0, s, c->counters, c->cand_cap,
             reinterpret_cast<unsigned long long *>(counts), c->status);
  p3t_note_launches(2);
  (void)p;
  return cudaGetLastError() == cudaSuccess ? P3T_OK : P3T_ERR_CUDA;
}

// entries of a walk's stack in a context of up to n particles: all that can stand
// there.  A warp pops the deepest 32 and pushes their children in the same order,
// so the stack's levels ascend: a level's nodes are opened only when all deeper
// ones are among the popped, so at most 8 x 32 entries of a level stand there (the
// first two levels 8 and 64), and as disjoint subtrees no more than the particles.
// (Disks of 1e3 to 1e6 bodies reach 70 to 464.)
int64_t p3t_walk_stack(int64_t n) {
  return std::min<int64_t>(n, 8 + 64 + 256 * (P3T_BITS - 2));
}

// persistent walk warps for a context of up to n particles: the most blocks per SM
// of the kernels that take it (a program may hold many small contexts: 5,000 bodies
// 122 -> 55 MB each), fewer still below: a block for every 4 particles (the FP64 walks take
// single targets there; with a block for every 256, 1,000 particles in FP64
// ran on 4 SMs: 2,535 us at theta = 0, 105 now; mixed 1e5 ring 338 -> 253)
int64_t p3t_walk_warps(int num_sms, int64_t n) {
  const bool small = n <= (int64_t)kFewTargets * num_sms;
  int64_t blocks = (int64_t)num_sms * (small ? std::max(kWalk64Blocks, kFewBlocks) : kManyBlocks);
  const int64_t want = n / 4 + 1;
  if (want < blocks) blocks = want;
  return blocks * kWarps;
}
