// Soft step: neighbour lists and neighbour clusters
// (Sec. 2.3).  Compiled with -fmad=false: the neighbour predicate is decided
// in FP64 with a fixed evaluation order so that membership is bit-exact.
#include "block_sort.cuh"
#include "p3t_internal.cuh"

namespace {

constexpr int kBlock = 256;
constexpr int64_t kUFLimit = 1 << 26;  // bound on union-find retries per edge

// Sec. 2.3: candidate j of i (r_ij < max(r_search,i, r_search,j)) stays a
// neighbour iff the closest approach of the linear relative motion over
// [0, dt] (Eq. rsearch1 with the clamped t_min) is within R~s,2 r_out,ij, or
// v_ij < R~s,3 a_ij dt/2 with a_ij = G (m_i + m_j) / r_ij^2.
__device__ __forceinline__ bool neighbour_pair(int32_t i, int32_t j,
                                               const p3t_particles &p,
                                               const p3t_params &prm) {
  const double rx = p.x[i] - p.x[j], ry = p.y[i] - p.y[j], rz = p.z[i] - p.z[j];
  const double r2 = rx * rx + ry * ry + rz * rz;
  const double rs = fmax(p.r_search[i], p.r_search[j]);
  if (!(r2 < rs * rs)) return false;
  const double ux = p.vx[i] - p.vx[j], uy = p.vy[i] - p.vy[j], uz = p.vz[i] - p.vz[j];
  const double v2 = ux * ux + uy * uy + uz * uz;
  const double rv = rx * ux + ry * uy + rz * uz;
  double t = 0.0;
  if (v2 > 0.0) {
    t = -rv / v2;
    if (t < 0.0) t = 0.0;
    if (t >= prm.dt_soft) t = prm.dt_soft;
  }
  const double dx = rx + ux * t, dy = ry + uy * t, dz = rz + uz * t;
  const double d2 = dx * dx + dy * dy + dz * dz;
  const double lim = prm.rs2 * fmax(p.r_out[i], p.r_out[j]);
  if (d2 <= lim * lim) return true;
  const double a = prm.G * (p.m[i] + p.m[j]) / r2;
  const double w = prm.rs3 * a * prm.dt_soft * 0.5;
  return v2 < w * w;
}

__global__ void k_nb_filter(const int64_t *d_ncand, const int32_t *cand_i,
                            const int32_t *cand_j, const int32_t *idx,
                            const p3t_particles p, const p3t_params prm,
                            int32_t *keep, int32_t *deg, const DevStatus *st) {
  pdl_wait();
  if (st->code != 0) return;
  const int64_t nc = *d_ncand;
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < nc;
       k += (int64_t)gridDim.x * blockDim.x) {
    const int32_t i = idx[cand_i[k]], j = idx[cand_j[k]];
    const bool ok = neighbour_pair(i, j, p, prm);
    keep[k] = ok ? 1 : 0;
    if (ok) atomicAdd(&deg[i], 1);
  }
}

// the kept candidates into their rows (in any order; deg counts down to zero).
// A total above the capacity is recorded and nothing is written
__global__ void k_nb_fill(const int64_t *d_ncand, const int32_t *cand_i,
                          const int32_t *cand_j, const int32_t *idx,
                          const int32_t *keep, const int64_t *nb_off, const int64_t *nb_total,
                          int64_t nb_cap, int32_t *deg, int32_t *nb_idx, DevStatus *st) {
  pdl_wait();
  if (*nb_total > nb_cap) {
    if (blockIdx.x == 0 && threadIdx.x == 0) dev_fail(st, P3T_ERR_CAPACITY, 50, *nb_total);
    return;
  }
  if (st->code != 0) return;
  const int64_t nc = *d_ncand;
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < nc;
       k += (int64_t)gridDim.x * blockDim.x) {
    if (!keep[k]) continue;
    const int32_t i = idx[cand_i[k]], j = idx[cand_j[k]];
    const int32_t q = atomicSub(&deg[i], 1) - 1;
    nb_idx[nb_off[i] + q] = j;
  }
}

// rows are short (<n_b> << 1 in the paper's runs): insertion sort per row; and
// the start of the union-find: every particle its own root, of one member
__global__ void k_nb_sort_rows(int64_t n, const int64_t *nb_off, int32_t *nb_idx,
                               int32_t *parent, int32_t *csize, int64_t *cl_counts,
                               unsigned long long *huge, const DevStatus *st) {
  pdl_wait();
  if (blockIdx.x == 0 && threadIdx.x < 4) cl_counts[threadIdx.x] = 0;
  if (blockIdx.x == 0 && threadIdx.x < 2) huge[threadIdx.x] = 0ull;
  const bool failed = st->code != 0;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    parent[i] = (int32_t)i;
    csize[i] = 1;
    if (failed) continue;
    const int64_t b = nb_off[i], e = nb_off[i + 1];
    for (int64_t u = b + 1; u < e; ++u) {
      const int32_t v = nb_idx[u];
      int64_t w = u - 1;
      while (w >= b && nb_idx[w] > v) { nb_idx[w + 1] = nb_idx[w]; --w; }
      nb_idx[w + 1] = v;
    }
  }
}

// ---- union-find: a root is the smallest index of its tree -----------------
__device__ __forceinline__ int32_t uf_find(const int32_t *parent, int32_t x) {
  int32_t p = __ldcg(&parent[x]);
  int64_t guard = 0;
  while (p != x && guard++ < kUFLimit) { x = p; p = __ldcg(&parent[x]); }
  return x;
}

__global__ void k_uf_union(int64_t n, const int64_t *nb_off, const int32_t *nb_idx,
                           int32_t *parent, DevStatus *st) {
  pdl_wait();
  if (st->code != 0) return;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    for (int64_t q = nb_off[i]; q < nb_off[i + 1]; ++q) {
      const int32_t j = nb_idx[q];
      if (j <= i) continue;
      int64_t tries = 0;
      for (;;) {
        int32_t a = uf_find(parent, (int32_t)i), b = uf_find(parent, j);
        if (a == b) break;
        if (a > b) { int32_t t = a; a = b; b = t; }
        // hook the larger root below the smaller one
        if (atomicCAS(&parent[b], b, a) == b) break;
        if (++tries > kUFLimit) { dev_fail(st, P3T_ERR_TIMEOUT, 51, 0); return; }
      }
    }
  }
}

// each particle's root, the clusters' sizes (a root counts itself from the start)
// and, from their counting, the others' places among their cluster's members (in
// any order).  A warp's members of one cluster are counted by one addition
__global__ void k_uf_label(int64_t n, const int32_t *parent, int32_t *label,
                           int32_t *csize, int32_t *place) {
  pdl_wait();
  const int lane = threadIdx.x & 31;
  for (int64_t i0 = blockIdx.x * (int64_t)blockDim.x + (threadIdx.x - lane); i0 < n;
       i0 += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = i0 + lane;
    int32_t r = -1;
    if (i < n) {
      r = uf_find(parent, (int32_t)i);
      label[i] = r;
      if (r == i) r = -1;
    }
    if (!__any_sync(0xffffffffu, r >= 0)) continue;
    const unsigned same = __match_any_sync(0xffffffffu, r);
    const int first = __ffs(same) - 1;
    int32_t at = 0;
    if (r >= 0 && lane == first) at = atomicAdd(&csize[r], __popc(same));
    at = __shfl_sync(0xffffffffu, at, first);
    if (r >= 0) place[i] = at + __popc(same & ((1u << lane) - 1u));
  }
}

// The members of every cluster in index order.  A cluster is a few members almost
// always, but close to percolation there are many of any size, so each size has
// a form of its own and consecutive clusters go to different blocks: a thread
// sorts up to eight members in registers, a warp ranks up to 32 and sorts up to
// 256, a block sorts up to kMemMax in shared memory.  Larger ones (at most n /
// kMemMax) are numbered and placed in order: the particles are cut into kSlices
// equal slices, k_cl_scatter counts each such cluster's members in each slice
// and sums the counts before, and a warp a slice then writes its members.
// Bound by its launch and the members' latency: equal-mass ring, N = 1e5, 4 us,
// wide disk, N = 1e6, 5; sorting all members by label took three radix passes and
// a copy, some 55 us in both.  The whole neighbour stage near percolation, with
// that sort, with one block for all clusters above 32 members, and now: 1,000
// clusters of 40 in 1e5 particles 100, 1,090, 71 us; 1,000 of 600 in 1e6 326,
// 8,600, 320; 900 of 1,030 457, 229,000, 434; one of 200,000 340, 740, 328.
constexpr int kMemThreads = 1024, kMemSmall = 8, kMemMax = kMemThreads * kItems;
constexpr int kSlices = 1024;
// the clusters above kMemMax: how many, the number of a root's cluster and, in the
// union-find's words (free by then, n of them), a row of kSlices counts each
struct Huge {
  unsigned long long *count;  // [1]: the blocks of k_cl_scatter done
  int32_t *number, *words;
  __device__ __forceinline__ int32_t *row(int64_t h) const { return words + h * kSlices; }
};
__device__ __forceinline__ int slice_len(int64_t n) { return (int)((n + kSlices - 1) / kSlices); }

// two flag words a particle: [0, n) isolated, member of a cluster; [n, 2n) root of
// a cluster and its size
__global__ void k_cl_flags(int64_t n, const int32_t *label, const int32_t *csize,
                           int32_t *flag, int64_t *counts, Huge huge) {
  pdl_wait();
  unsigned long long mx = 0;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    const int32_t sz = csize[label[i]];
    const bool root = label[i] == i && csize[i] >= 2;
    // two words a particle, each scanned as (bit 0) + (bits 1-31) 2^31:
    // isolated and cluster member; cluster root and its size
    flag[i] = (sz == 1 ? 1 : 0) | (sz >= 2 ? 2 : 0);
    flag[n + i] = root ? 1 | (csize[i] << 1) : 0;
    if (root) mx = max(mx, (unsigned long long)csize[i]);
  }
  if (mx) atomicMax(reinterpret_cast<unsigned long long *>(&counts[3]), mx);
  if (mx <= kMemMax) return;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    if (label[i] != i || csize[i] <= kMemMax) continue;
    const int64_t h = (int64_t)atomicAdd(huge.count, 1ull);
    huge.number[i] = (int32_t)h;
    int4 *row = reinterpret_cast<int4 *>(huge.row(h));
    for (int q = 0; q < kSlices / 4; ++q) row[q] = make_int4(0, 0, 0, 0);
  }
}

// the singles, each cluster's offset and its members (in any order, by their
// places) from the two packed scans (counts in bits 0-30, the second sum from
// bit 31), and the totals: singles, clusters, members (counts[0..2])
__global__ void k_cl_scatter(int64_t n, const int32_t *label, const int32_t *flag,
                             const int64_t *pos, const int64_t *d_tot, int32_t *singles,
                             int64_t *cl_off, const int32_t *place, int32_t *mem, int64_t *counts,
                             Huge huge) {
  pdl_wait();
  constexpr int64_t kLow = (1ll << 31) - 1;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    const int32_t fa = flag[i], fb = flag[n + i];
    if (fa & 1) singles[pos[i] & kLow] = (int32_t)i;
    if (fb & 1) {
      const int64_t q = pos[n + i];
      cl_off[q & kLow] = q >> 31;
    }
    if (fa & 2) {
      // (those of a cluster above kMemMax are counted by slice)
      const int32_t r = label[i];
      if ((flag[n + r] >> 1) <= kMemMax)
        mem[(pos[n + r] >> 31) + (r == i ? 0 : place[i])] = (int32_t)i;
      else
        atomicAdd(&huge.row(huge.number[r])[(int)i / slice_len(n)], 1);
    }
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    const int64_t ta = d_tot[0], tb = d_tot[1];
    counts[0] = ta & kLow;
    counts[1] = tb & kLow;
    counts[2] = tb >> 31;
    cl_off[tb & kLow] = tb >> 31;
  }
  const int64_t nh = (int64_t)*huge.count;
  if (nh == 0) return;
  // the last block to finish: each row of counts to the sums of those before
  __threadfence();
  __syncthreads();
  if (!__syncthreads_or(threadIdx.x == 0 && atomicAdd(&huge.count[1], 1ull) == gridDim.x - 1))
    return;
  __threadfence();
  const int lane = threadIdx.x & 31;
  for (int64_t h = threadIdx.x >> 5; h < nh; h += blockDim.x >> 5) {
    int32_t *row = huge.row(h);
    int run = 0;
    for (int q = lane; q < kSlices; q += 128) {
      int c[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) c[k] = __ldcg(&row[q + 32 * k]);
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        int v = c[k];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const int u = __shfl_up_sync(0xffffffffu, v, o);
          if (lane >= o) v += u;
        }
        row[q + 32 * k] = run + v - c[k];
        run += __shfl_sync(0xffffffffu, v, 31);
      }
    }
  }
}

// the members of the clusters above kMemMax, a warp a slice of the particles (its
// cluster's word of the row is the warp's own)
__device__ void place_huge(int64_t n, const Huge &huge, const int32_t *label, const int32_t *flag,
                           const int64_t *pos, int32_t *mem) {
  const int lane = threadIdx.x & 31, len = slice_len(n);
  const int64_t warps = (int64_t)gridDim.x * (kMemThreads / 32);
  // neighbouring slices to different blocks
  for (int64_t sl = blockIdx.x + (int64_t)gridDim.x * (threadIdx.x >> 5); sl < kSlices;
       sl += warps) {
    const int64_t i0 = sl * len, i1 = min(n, i0 + len);
    constexpr int kRows = 4;  // rows of 32 whose loads are in flight together
    for (int64_t b = i0; b < i1; b += 32 * kRows) {
      int32_t r[kRows], h[kRows];
      int64_t o[kRows];
#pragma unroll
      for (int k = 0; k < kRows; ++k) {
        const int64_t i = b + 32 * k + lane;
        r[k] = i < i1 ? label[i] : -1;
      }
#pragma unroll
      for (int k = 0; k < kRows; ++k) {
        const bool on = r[k] >= 0 && (flag[n + r[k]] >> 1) > kMemMax;
        h[k] = on ? huge.number[r[k]] : -1;
        o[k] = on ? pos[n + r[k]] >> 31 : 0;
      }
#pragma unroll
      for (int k = 0; k < kRows; ++k) {
        const unsigned same = __match_any_sync(0xffffffffu, h[k]);
        const int first = __ffs(same) - 1;
        int32_t at = 0;
        if (h[k] >= 0 && lane == first) at = atomicAdd(&huge.row(h[k])[sl], __popc(same));
        at = __shfl_sync(0xffffffffu, at, first);
        if (h[k] >= 0)
          mem[o[k] + at + __popc(same & ((1u << lane) - 1u))] = (int32_t)(b + 32 * k + lane);
      }
    }
  }
}

__global__ void __launch_bounds__(kMemThreads) k_cl_sort(const int64_t *counts,
                                                         const int64_t *cl_off, int64_t n,
                                                         const int32_t *label, const int32_t *flag,
                                                         const int64_t *pos, int32_t *mem,
                                                         Huge huge) {
  pdl_wait();
  __shared__ uint32_t s_mem[kMemMax + kMemMax / 8];
  __shared__ int s_list[2][kMemThreads], s_n[2];  // clusters for a warp, for the block
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int64_t ncl = counts[1], nh = (int64_t)*huge.count;
  // clusters b, b + gridDim, b + 2 gridDim, ... to block b
  for (int64_t t0 = 0; blockIdx.x + gridDim.x * t0 < ncl; t0 += kMemThreads) {
    if (threadIdx.x < 2) s_n[threadIdx.x] = 0;
    __syncthreads();
    const int64_t c = blockIdx.x + gridDim.x * (t0 + threadIdx.x);
    if (c < ncl) {
      const int64_t o = cl_off[c];
      const int m = (int)(cl_off[c + 1] - o);
      if (m <= kMemSmall) {
        int32_t v[kMemSmall];
#pragma unroll
        for (int k = 0; k < kMemSmall; ++k) v[k] = k < m ? mem[o + k] : 0x7fffffff;
        // odd-even transposition, as many rounds as members
#pragma unroll
        for (int r = 0; r < kMemSmall; ++r) {
          if (r < m)
#pragma unroll
            for (int k = r & 1; k + 1 < kMemSmall; k += 2) {
              const int32_t lo = min(v[k], v[k + 1]), hi = max(v[k], v[k + 1]);
              v[k] = lo;
              v[k + 1] = hi;
            }
        }
#pragma unroll
        for (int k = 0; k < kMemSmall; ++k)
          if (k < m) mem[o + k] = v[k];
      } else if (m <= kMemMax) {
        const int q = m > 32 * kItems;
        s_list[q][atomicAdd(&s_n[q], 1)] = threadIdx.x;
      }
    }
    __syncthreads();
    for (int q = w; q < s_n[0]; q += kMemThreads / 32) {
      const int64_t d = blockIdx.x + gridDim.x * (t0 + s_list[0][q]), o = cl_off[d];
      const int m = (int)(cl_off[d + 1] - o);
      if (m <= 32) {
        const int32_t v = lane < m ? mem[o + lane] : 0x7fffffff;
        int rank = 0;
        for (int j = 0; j < m; ++j) rank += __shfl_sync(0xffffffffu, v, j) < v;
        if (lane < m) mem[o + rank] = v;
      } else {
        uint32_t v[kItems];
#pragma unroll
        for (int k = 0; k < kItems; ++k)
          v[k] = 32 * k + lane < m ? (uint32_t)mem[o + 32 * k + lane] : ~0u;
        warp_sort(v);
#pragma unroll
        for (int k = 0; k < kItems; ++k)
          if (kItems * lane + k < m) mem[o + kItems * lane + k] = (int32_t)v[k];
      }
    }
    for (int q = 0; q < s_n[1]; ++q) {
      const int64_t d = blockIdx.x + gridDim.x * (t0 + s_list[1][q]), o = cl_off[d];
      const int m = (int)(cl_off[d + 1] - o);
      for (int e = threadIdx.x; e < m; e += kMemThreads) s_mem[slot(e)] = (uint32_t)mem[o + e];
      __syncthreads();
      sort_words(s_mem, m);
      for (int e = threadIdx.x; e < m; e += kMemThreads) mem[o + e] = (int32_t)s_mem[slot(e)];
      __syncthreads();
    }
    __syncthreads();
  }
  if (nh > 0) place_huge(n, huge, label, flag, pos, mem);
}

}  // namespace

int p3t_run_neighbours(p3t_ctx *c, const p3t_particles *p, int64_t *nb_off,
                       int32_t *nb_idx, int64_t nb_cap, cudaStream_t s) {
  const int64_t n = p->n;
  const int64_t maxb = (int64_t)c->num_sms * P3T_NSM_BLOCKS;
  const int64_t g = p3t_grid(n, kBlock, maxb);
  const int64_t gc = p3t_grid(c->cand_cap, kBlock, maxb);
  int64_t *cnt = c->counters;
  int rc;
  // (counters[28], [29]; the rows' degrees are spent when the roots are numbered;
  // the third quarter of the flags holds the places)
  const Huge huge{reinterpret_cast<unsigned long long *>(&cnt[28]), c->deg, c->parent};
  int32_t *place = c->flag + 2 * c->cap;
  // ---- neighbour lists ----
  P3T_CUDA_TRY(cudaMemsetAsync(c->deg, 0, sizeof(int32_t) * (n + 1), s));
  pdl_launch(k_nb_filter, dim3((unsigned)gc), dim3(kBlock), 0, s, &cnt[9], c->cand_i, c->cand_j, c->idx, *p,
                                              c->prm, c->cand_keep, c->deg, c->status);
  rc = p3t_scan_i32_to_i64(c->deg, nb_off, &cnt[0], c->cap, nb_off + n, c->scan_state, c->scan_words, c->status, c->poll_limit, s);
  if (rc) return rc;
  pdl_launch(k_nb_fill, dim3((unsigned)gc), dim3(kBlock), 0, s, &cnt[9], c->cand_i, c->cand_j,
             c->idx, c->cand_keep, nb_off, nb_off + n, nb_cap, c->deg, nb_idx, c->status);
  pdl_launch(k_nb_sort_rows, dim3((unsigned)g), dim3(kBlock), 0, s, n, nb_off, nb_idx, c->parent,
             c->csize, c->cl_counts, huge.count, c->status);
  // ---- neighbour clusters ----
  pdl_launch(k_uf_union, dim3((unsigned)g), dim3(kBlock), 0, s, n, nb_off, nb_idx, c->parent, c->status);
  pdl_launch(k_uf_label, dim3((unsigned)g), dim3(kBlock), 0, s, n, c->parent, c->label, c->csize, place);
  pdl_launch(k_cl_flags, dim3((unsigned)g), dim3(kBlock), 0, s, n, c->label, c->csize, c->flag, c->cl_counts, huge);
  // two packed scans: (isolated, members) and (roots, root sizes); their
  // totals in cnt[21], cnt[22]
  for (int q = 0; q < 2; ++q) {
    rc = p3t_scan_flag_pairs(c->flag + q * n, c->pos + q * n, &cnt[0], c->cap, &cnt[21 + q],
                             c->scan_state, c->scan_words, c->status, c->poll_limit, s);
    if (rc) return rc;
  }
  // the members stay in one buffer, so that the cluster views keep their
  // addresses from step to step (a step captured in a CUDA graph reads the
  // previous step's clusters there)
  pdl_launch(k_cl_scatter, dim3((unsigned)g), dim3(kBlock), 0, s, n, c->label, c->flag, c->pos,
             &cnt[21], c->singles, c->cl_off, place, c->mvals, c->cl_counts, huge);
  pdl_launch(k_cl_sort, dim3((unsigned)p3t_grid(n / 2 + 1, kMemThreads, c->num_sms)), dim3(kMemThreads), 0,
             s, c->cl_counts, c->cl_off, n, c->label, c->flag, c->pos, c->mvals, huge);
  // filter, fill, sort_rows, uf_union, uf_label, flags, scatter, sort
  p3t_note_launches(8);
  c->cl_mem = c->mvals;
  return cudaGetLastError() == cudaSuccess ? P3T_OK : P3T_ERR_CUDA;
}
