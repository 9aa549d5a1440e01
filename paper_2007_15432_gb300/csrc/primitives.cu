// Device-wide primitives of libp3t: exclusive scan and stable LSD radix sort.
// Element counts are read from device memory so that a whole soft step can be
// enqueued (and captured in a CUDA graph) without reading sizes on the host.
#include "block_sort.cuh"
#include "p3t_internal.cuh"

namespace {

__device__ __forceinline__ int64_t warp_incl_scan(int64_t v) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    int64_t t = __shfl_up_sync(0xffffffffu, v, o);
    if (lane >= o) v += t;
  }
  return v;
}

// block-wide exclusive scan of one value per thread; returns the block total
__device__ int64_t block_excl_scan(int64_t v, int64_t *excl, int64_t *sh) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
  int64_t inc = warp_incl_scan(v);
  if (lane == 31) sh[w] = inc;
  __syncthreads();
  if (w == 0) {
    int64_t s = lane < nw ? sh[lane] : 0;
    int64_t si = warp_incl_scan(s);
    if (lane < nw) sh[lane] = si - s;
    if (lane == 31) sh[32] = si;
  }
  __syncthreads();
  *excl = inc - v + sh[w];
  int64_t tot = sh[32];
  __syncthreads();
  return tot;
}

// ---- single-pass exclusive scan (decoupled look-back) -----------------------
// Each block takes the next tile number from a counter in state[0] (so every
// smaller tile belongs to a block that has started and will finish without
// waiting on this one), scans its tile, publishes the tile's sum, adds its
// predecessors' sums by looking back (a warp reads 32 predecessor words at a
// time and stops at the nearest one that holds an inclusive prefix), and
// publishes its own inclusive prefix.  A word holds a flag in bits 63-62 (1:
// the tile's own sum, 2: inclusive prefix) and the value in bits 61-0
// (non-negative inputs).  The grid is sized for the capacity; only as many
// blocks as the count has tiles take one, the rest return at once.  The last
// block to finish (counter state[1]) clears the words it used and both
// counters, so that the next call starts clean with no host involvement.  A bounded number of polls: a predecessor that
// never publishes is reported (P3T_ERR_TIMEOUT) and counted as zero.  With
// PAIRS, every input holds a 0/1 flag in bit 0 and a non-negative value in
// bits 1-31 and counts as flag + value 2^31, so that one scan gives both
// prefix sums (each below 2^31) in one word.
constexpr int kScanThreads = 512;
constexpr int kScanPer = 8;
constexpr int kScanTile = kScanThreads * kScanPer;
constexpr unsigned long long kFlagAgg = 1ull << 62, kFlagInc = 2ull << 62;
constexpr unsigned long long kValMask = (1ull << 62) - 1;
template <bool PAIRS>
__device__ __forceinline__ int64_t scan_value(int32_t v) {
  return PAIRS ? (int64_t)(v & 1) + ((int64_t)((uint32_t)v >> 1) << 31) : (int64_t)v;
}
template <bool PAIRS>
__global__ void __launch_bounds__(kScanThreads)
scan_onepass(const int32_t *in, int64_t *out, const int64_t *d_n, int64_t *d_total,
             unsigned long long *state, DevStatus *st, int64_t poll_limit) {
  pdl_wait();
  __shared__ int64_t sh[33];
  // the tile: first its int32 inputs, then its int64 outputs (staged so that
  // both the loads and the stores are coalesced)
  __shared__ __align__(16) int64_t s_buf[kScanTile];
  int32_t *s_in = reinterpret_cast<int32_t *>(s_buf);
  __shared__ unsigned long long s_tile;
  __shared__ int64_t s_prefix;
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const int64_t n = *d_n;
  // the grid is sized for the capacity: only the first `used` blocks take
  // tiles (and count themselves out below); the others return at once
  const int64_t used = (n + kScanTile - 1) / kScanTile;
  const int64_t takers = used < 1 ? 1 : (used < (int64_t)gridDim.x ? used : (int64_t)gridDim.x);
  if ((int64_t)blockIdx.x >= takers) return;
  const bool alone = used <= 1;  // one tile: no look-back, no state
  if (t == 0) s_tile = alone ? 0ull : atomicAdd(&state[0], 1ull);
  __syncthreads();
  const int64_t tile = (int64_t)s_tile;
  const int64_t base = tile * kScanTile;
  unsigned long long *ts = state + 2;
  if (base < n) {
    for (int i = 0; i < kScanPer; ++i) {
      const int64_t e = base + (int64_t)i * kScanThreads + t;
      s_in[i * kScanThreads + t] = e < n ? in[e] : 0;
    }
    __syncthreads();
    int32_t v[kScanPer];
    int64_t sum = 0;
    {
      const int4 a = reinterpret_cast<const int4 *>(s_in)[2 * t];
      const int4 b = reinterpret_cast<const int4 *>(s_in)[2 * t + 1];
      v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
      v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
    }
#pragma unroll
    for (int i = 0; i < kScanPer; ++i) sum += scan_value<PAIRS>(v[i]);
    int64_t ex;
    const int64_t agg = block_excl_scan(sum, &ex, sh);
    if (warp == 0) {
      int64_t prefix = 0;
      if (tile == 0) {
        if (lane == 0 && !alone) {
          __threadfence();
          __stcg(&ts[0], kFlagInc | (unsigned long long)agg);
        }
      } else {
        if (lane == 0) {
          __threadfence();
          __stcg(&ts[tile], kFlagAgg | (unsigned long long)agg);
        }
        int64_t p = tile - 1;  // the window's first (nearest) predecessor
        int64_t polls = 0;
        for (;;) {
          const int64_t q = p - lane;
          unsigned long long w = q >= 0 ? __ldcv(&ts[q]) : kFlagInc;
          while (__any_sync(0xffffffffu, (w >> 62) == 0)) {
            if (++polls > poll_limit) {
              if (lane == 0) dev_fail(st, P3T_ERR_TIMEOUT, 70, 0);
              w = (w >> 62) == 0 ? kFlagAgg : w;  // count the silent tile as zero
              break;
            }
            __nanosleep(64);
            if ((w >> 62) == 0) w = __ldcv(&ts[q]);
          }
          const unsigned inc = __ballot_sync(0xffffffffu, (w >> 62) == 2);
          const int last = inc ? __ffs(inc) - 1 : 31;  // nearest inclusive prefix
          int64_t val = lane <= last ? (int64_t)(w & kValMask) : 0;
          for (int o = 16; o > 0; o >>= 1) val += __shfl_xor_sync(0xffffffffu, val, o);
          prefix += val;
          if (inc) break;
          p -= 32;
        }
        if (lane == 0) {
          __threadfence();
          __stcg(&ts[tile], kFlagInc | (unsigned long long)(prefix + agg));
        }
      }
      if (lane == 0) s_prefix = prefix;
    }
    __syncthreads();  // every thread has read its inputs: s_buf now holds outputs
    int64_t run = s_prefix + ex;
#pragma unroll
    for (int i = 0; i < kScanPer; ++i) {
      s_buf[t * kScanPer + i] = run;
      run += scan_value<PAIRS>(v[i]);
    }
    __syncthreads();
    for (int i = 0; i < kScanPer; ++i) {
      const int64_t e = base + (int64_t)i * kScanThreads + t;
      if (e < n) out[e] = s_buf[i * kScanThreads + t];
    }
    if (t == 0 && base + kScanTile >= n && d_total) *d_total = s_prefix + agg;
  } else if (t == 0 && tile == 0 && d_total) {
    *d_total = 0;  // n = 0
  }
  if (alone) return;
  // the last block out resets the tile words and the counters
  __shared__ bool s_last;
  __syncthreads();
  if (t == 0) {
    __threadfence();
    s_last = atomicAdd(&state[1], 1ull) == (unsigned long long)takers - 1;
  }
  __syncthreads();
  if (s_last) {
    __threadfence();
    for (int64_t k = t; k < used; k += kScanThreads) ts[k] = 0ull;
    if (t == 0) { state[0] = 0ull; state[1] = 0ull; }
  }
}

// ---- radix sort -----------------------------------------------------------
constexpr int kRadixBits = 8;
constexpr int kRadix = 1 << kRadixBits;
constexpr int kSortThreads = 256;
constexpr int kSortItems = 8;
constexpr int kSortTile = kSortThreads * kSortItems;

// The grids are sized for the capacity; the tiles actually holding keys
// (from the count on the device) are dealt grid-stride, so a short sort (a
// few thousand cluster members in a buffer sized for every particle) costs
// little more than its launches.  hist rows keep the capacity's stride.
__device__ __forceinline__ int64_t radix_tiles(const int64_t *d_n) {
  return (*d_n + kSortTile - 1) / kSortTile;
}

__global__ void radix_upsweep(const uint64_t *keys, const int64_t *d_n,
                              int shift, uint32_t *hist, int ntiles) {
  pdl_wait();
  __shared__ uint32_t h[kRadix];
  const int64_t n = *d_n;
  const int64_t used = radix_tiles(d_n);
  for (int64_t tile = blockIdx.x; tile < used; tile += gridDim.x) {
    h[threadIdx.x] = 0;
    __syncthreads();
    const int64_t base = tile * kSortTile;
    // every load of the tile issued before the first is used
    uint32_t dig[kSortItems];
#pragma unroll
    for (int k = 0; k < kSortItems; ++k) {
      const int64_t e = base + k * kSortThreads + threadIdx.x;
      dig[k] = e < n ? (uint32_t)((__ldg(&keys[e]) >> shift) & (kRadix - 1)) : kRadix;
    }
    // plain shared atomics: on this part a warp's same-address atomics cost
    // less than matching the lanes' digits first
#pragma unroll
    for (int k = 0; k < kSortItems; ++k)
      if (dig[k] < kRadix) atomicAdd(&h[dig[k]], 1u);
    __syncthreads();
    hist[(int64_t)threadIdx.x * ntiles + tile] = h[threadIdx.x];
    __syncthreads();
  }
}

// exclusive scan of each digit's row of tile counts (one block per digit);
// the row total goes to the last slot of the digit's totals
__global__ void __launch_bounds__(kRadix) radix_row_scan(uint32_t *hist, int ntiles,
                                                         uint32_t *digit_total,
                                                         const int64_t *d_n) {
  pdl_wait();
  __shared__ int64_t sh[33];
  uint32_t *row = hist + (int64_t)blockIdx.x * ntiles;
  const int used = (int)radix_tiles(d_n);
  int64_t carry = 0;
  for (int base = 0; base < used; base += kRadix) {
    const int i = base + threadIdx.x;
    const int64_t v = i < used ? row[i] : 0;
    int64_t ex;
    const int64_t tot = block_excl_scan(v, &ex, sh);
    if (i < used) row[i] = (uint32_t)(carry + ex);
    carry += tot;
  }
  if (threadIdx.x == 0) digit_total[blockIdx.x] = (uint32_t)carry;
}

// The lanes of the warp whose (valid) digit equals this lane's: eight ballots,
// one a bit of the digit (on this part cheaper than __match_any_sync); zero
// for an invalid lane
__device__ __forceinline__ uint32_t match_digit(uint32_t d, bool valid) {
  uint32_t m = __ballot_sync(0xffffffffu, valid);
#pragma unroll
  for (int b = 0; b < kRadixBits; ++b) {
    const uint32_t bb = __ballot_sync(0xffffffffu, (d >> b) & 1u);
    m &= ((d >> b) & 1u) ? bb : ~bb;
  }
  return valid ? m : 0u;
}

// Stable scatter of one tile: the tile's elements are ranked by (digit,
// position), placed digit-ordered in shared memory, then written out so that
// consecutive threads write consecutive addresses of one digit's run.
__global__ void __launch_bounds__(kSortThreads)
radix_downsweep(const uint64_t *keys, const int32_t *vals, uint64_t *okeys,
                int32_t *ovals, const int64_t *d_n, int shift,
                const uint32_t *hist, int ntiles, const uint32_t *digit_total, int32_t *inv) {
  pdl_wait();
  __shared__ uint32_t s_warp[kSortThreads / 32][kRadix];
  __shared__ uint32_t s_run[kRadix];
  __shared__ uint32_t s_gbase[kRadix];  // first output index of the tile's digit d
  __shared__ uint32_t s_lbase[kRadix];  // first tile position of digit d
  __shared__ int64_t sh[33];
  __shared__ uint64_t s_key[kSortTile];
  __shared__ int32_t s_val[kSortTile];
  const int t = threadIdx.x, lane = t & 31, w = t >> 5;
  const int64_t n = *d_n;
  const int64_t used = radix_tiles(d_n);
  if (blockIdx.x >= used) return;  // no tile of this sort for this block
  int64_t dbase;
  block_excl_scan((int64_t)digit_total[t], &dbase, sh);   // digit bases
  for (int64_t tile = blockIdx.x; tile < used; tile += gridDim.x) {
    __syncthreads();
    s_run[t] = 0;
    s_gbase[t] = (uint32_t)dbase + hist[(int64_t)t * ntiles + tile];
    const int64_t base = tile * kSortTile;
    const uint32_t lt = (1u << lane) - 1u;
    uint64_t key[kSortItems];
    int32_t val[kSortItems];
    uint32_t dig[kSortItems], rk[kSortItems];
    // the tile's loads all issued up front: the ranking rounds below are
    // separated by block barriers, which no load can be moved across
#pragma unroll
    for (int r = 0; r < kSortItems; ++r) {
      const int64_t e = base + r * kSortThreads + t;
      key[r] = 0;
      val[r] = 0;
      if (e < n) {
        key[r] = __ldg(&keys[e]);
        val[r] = __ldg(&vals[e]);
      }
    }
#pragma unroll
    for (int r = 0; r < kSortItems; ++r) {
#pragma unroll
      for (int k = 0; k < kSortThreads / 32; ++k) s_warp[k][t] = 0;
      __syncthreads();
      const int64_t e = base + r * kSortThreads + t;
      const bool valid = e < n;
      // invalid lanes belong to no group
      const uint32_t d = valid ? (uint32_t)((key[r] >> shift) & (kRadix - 1)) : kRadix;
      dig[r] = d;
      const uint32_t peers = match_digit(d, valid);
      if (valid && lane == __ffs(peers) - 1) s_warp[w][d] = __popc(peers);
      __syncthreads();
      {
        uint32_t run = s_run[t];
#pragma unroll
        for (int k = 0; k < kSortThreads / 32; ++k) {
          uint32_t c = s_warp[k][t];
          s_warp[k][t] = run;
          run += c;
        }
        s_run[t] = run;
      }
      __syncthreads();
      rk[r] = valid ? s_warp[w][d] + __popc(peers & lt) : 0;  // rank within the tile's digit
      __syncthreads();
    }
    {
      int64_t ex;
      block_excl_scan((int64_t)s_run[t], &ex, sh);
      s_lbase[t] = (uint32_t)ex;
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < kSortItems; ++r)
      if (dig[r] < kRadix) {
        const uint32_t pos = s_lbase[dig[r]] + rk[r];
        s_key[pos] = key[r];
        s_val[pos] = val[r];
      }
    __syncthreads();
    const int64_t tn = n - base < kSortTile ? n - base : kSortTile;
    for (int i = t; i < tn; i += kSortThreads) {
      const uint64_t k = s_key[i];
      const uint32_t d = (uint32_t)((k >> shift) & (kRadix - 1));
      const uint32_t dst = s_gbase[d] + ((uint32_t)i - s_lbase[d]);
      okeys[dst] = k;
      ovals[dst] = s_val[i];
      if (inv) inv[s_val[i]] = (int32_t)dst;
    }
  }
}

// ---- sort by (key, value) ----------------------------------------------------
// The sorts of the library order distinct values by (key, value) (the values
// are indices that start in ascending order, so this is the stable order by
// key).  A radix pass is three launches whose tiles leave the chip waiting on
// L2 latency: 22 us at a million keys, 12 at three thousand, eight passes a
// tree.  Up to kSampleMax keys are sorted instead
//  - by one block in shared memory when the capacity is at most
//    kBlockSortMax (one launch);
//  - else as a sample sort: one block sorts 8 samples a bucket (4 with the most
//    buckets), at random positions of the input, and takes every eighth (fourth)
//    as a splitter, so that the buckets are balanced whatever the keys'
//    distribution and order: about 1,000 a bucket, and one above the 4,096 a
//    block holds has odds of 3e-8 (5e-5; it costs a merge of two runs, some 10
//    us; only an input made for these positions has larger ones), a pass finds
//    each key's bucket and its place in it (by atomics: the order within a
//    bucket is left to its sort), a pass moves it there, and a block sorts each
//    bucket.  Four launches.
// The order is unique, so the result is that of the radix passes.  Keys and
// values end in the buffers they started in.  Measured (mixed tree build): N =
// 1e6 381 -> 339 us, 1e5 200 -> 155, 3,001 178 -> 120, 1,000 (FP64) 200 -> 141.
// What bounds it: the one block that sorts the samples and the latency of the
// buckets' blocks (three of 512 threads an SM beat two, and blocks of 256 with
// buckets of 2,048: 339, 348, 346 us).  Keys of 32 bits or less keep the radix
// passes (cut-off bins of 377,740: 40 against 76 us).
constexpr int kBlockSortMax = 1024 * kItems;
static_assert(kBlockSortMax == P3T_SORT_BLOCK, "one block's sort");
constexpr int kLocalThreads = 512;
constexpr int kLocalMax = kLocalThreads * kItems;
constexpr int kMaxBuckets = 1024;
constexpr int kSamples = 4096;            // 8 a bucket, 4 of the most buckets
constexpr int64_t kSampleMax = 1500000;
constexpr int kPosBits = 21;              // place in a bucket: below kSampleMax < 2^21
constexpr int kPlace = 13;                // place in a block's input, below 2^13

struct SortWork {
  uint64_t skey[kMaxBuckets];
  int32_t sval[kMaxBuckets];
  uint32_t count[kMaxBuckets], start[kMaxBuckets + 1];
  int32_t done;
};

__device__ __forceinline__ bool pair_less(uint64_t ka, int32_t va, uint64_t kb, int32_t vb) {
  return ka < kb || (ka == kb && va < vb);
}
constexpr size_t sort_smem(int max) { return (size_t)(max + max / 8) * 12; }

// One 64-bit word per entry: the leading bits of its key (kb bits, taken
// relative to the smallest possible one), as much of its value (vb bits) as
// there is room for, and its place in the input.  Words order as (key, value)
// except among entries that agree in the whole upper part while something was
// cut off (exact() false).
struct WordSpec {
  int kb, vb;
  __device__ __forceinline__ bool exact() const { return kb + vb <= 64 - kPlace; }
  __device__ __forceinline__ uint64_t word(uint64_t key, int32_t val, int place) const {
    const int room = 64 - kPlace;
    uint64_t u;
    if (kb >= room) {
      u = key >> (kb - room);
    } else {
      const int w = min(vb, room - kb);
      u = (key << w) | (uint64_t)((uint32_t)val >> (vb - w));
    }
    return u << kPlace | (uint64_t)place;
  }
};

// entries [0, n) of (sk, sv) sorted by (key, value) in merge rounds: the plain
// form for entries that sort_words cannot tell apart
__device__ __noinline__ void block_sort(uint64_t *sk, int32_t *sv, int n) {
  const int i0 = threadIdx.x * kItems;
  const bool in = i0 < n;
  uint64_t k[kItems];
  int32_t v[kItems];
  for (int w = 1; w < n; w <<= 1) {
    if (in) {
      int last = -1, ia = 0, ib = 0, a1 = 0, b1 = 0;
      for (int q = 0; q < kItems && i0 + q < n; ++q) {
        const int base = (i0 + q) & ~(2 * w - 1);
        if (base != last) {
          const int diag = i0 + q - base;
          last = base;
          a1 = min(base + w, n);
          b1 = min(base + 2 * w, n);
          int lo = max(0, diag - (b1 - a1)), hi = min(diag, a1 - base);
          while (lo < hi) {
            const int mid = (lo + hi) >> 1;
            const int pa = slot(base + mid), pb = slot(a1 + diag - 1 - mid);
            if (pair_less(sk[pa], sv[pa], sk[pb], sv[pb])) lo = mid + 1; else hi = mid;
          }
          ia = base + lo;
          ib = a1 + diag - lo;
        }
        const bool ta = ib >= b1 || (ia < a1 && pair_less(sk[slot(ia)], sv[slot(ia)],
                                                          sk[slot(ib)], sv[slot(ib)]));
        const int f = slot(ta ? ia++ : ib++);
        k[q] = sk[f];
        v[q] = sv[f];
      }
    }
    __syncthreads();
    if (in)
      for (int q = 0; q < kItems && i0 + q < n; ++q) {
        sk[slot(i0 + q)] = k[q];
        sv[slot(i0 + q)] = v[q];
      }
    __syncthreads();
  }
}

// n entries of (ik, iv) (at most eight a thread) sorted into (ok, ov), which
// may be the same arrays; keys are at least lo and below lo + 2^kb.  With ok
// null the result stays in shared memory (*sk, *sv in slots).
__device__ void sort_entries(const uint64_t *ik, const int32_t *iv, uint64_t *ok, int32_t *ov,
                             int n, uint64_t lo, int kb, int vb, uint64_t *sk, int32_t *sv) {
  const WordSpec ws{kb, vb};
  const int t = threadIdx.x, nt = blockDim.x;
  for (int i = t; i < n; i += nt) sk[slot(i)] = ws.word(ik[i] - lo, iv[i], i);
  __syncthreads();
  sort_words(sk, n);
  // entries whose words agree but for the place: short runs (two bodies in a
  // cell) put in order here, longer ones by the plain sort
  bool bad = false;
  if (!ws.exact()) {
    for (int i = t; i < n; i += nt) {
      const uint64_t w = sk[slot(i)] >> kPlace;
      if (i > 0 && sk[slot(i - 1)] >> kPlace == w) continue;
      int e = i + 1;
      while (e < n && e - i <= 8 && sk[slot(e)] >> kPlace == w) ++e;
      if (e - i > 8) {
        bad = true;
      } else {
        for (int u = i + 1; u < e; ++u) {
          const uint64_t x = sk[slot(u)];
          const int px = (int)(x & ((1u << kPlace) - 1u));
          int z = u - 1;
          for (; z >= i; --z) {
            const uint64_t y = sk[slot(z)];
            const int py = (int)(y & ((1u << kPlace) - 1u));
            if (!pair_less(ik[px], iv[px], ik[py], iv[py])) break;
            sk[slot(z + 1)] = y;
          }
          sk[slot(z + 1)] = x;
        }
      }
    }
    if (__syncthreads_or(bad)) {
      for (int i = t; i < n; i += nt) { sk[slot(i)] = ik[i]; sv[slot(i)] = iv[i]; }
      __syncthreads();
      block_sort(sk, sv, n);
      if (ok)
        for (int i = t; i < n; i += nt) { ok[i] = sk[slot(i)]; ov[i] = sv[slot(i)]; }
      __syncthreads();
      return;
    }
  }
  uint64_t k[kItems];
  int32_t v[kItems];
#pragma unroll
  for (int q = 0; q < kItems; ++q) {
    const int i = t + q * nt;
    if (i < n) {
      const int p = (int)(sk[slot(i)] & ((1u << kPlace) - 1u));
      k[q] = ik[p];
      v[q] = iv[p];
    }
  }
  __syncthreads();
#pragma unroll
  for (int q = 0; q < kItems; ++q) {
    const int i = t + q * nt;
    if (i < n) {
      if (ok) { ok[i] = k[q]; ov[i] = v[q]; }
      else { sk[slot(i)] = k[q]; sv[slot(i)] = v[q]; }
    }
  }
  __syncthreads();
}

// up to kBlockSortMax entries, in place
__global__ void __launch_bounds__(1024) k_sort_block(uint64_t *keys, int32_t *vals,
                                                     const int64_t *d_n, int kb, int vb) {
  pdl_wait();
  extern __shared__ __align__(16) unsigned char sort_mem[];
  uint64_t *sk = reinterpret_cast<uint64_t *>(sort_mem);
  int32_t *sv = reinterpret_cast<int32_t *>(sk + kBlockSortMax + kBlockSortMax / 8);
  sort_entries(keys, vals, keys, vals, (int)*d_n, 0, kb, vb, sk, sv);
}

// Position of sample i of ns: a random one (i hashed by MurmurHash3's finalizer)
// in the i-th of ns strides.  (At the strides' starts the samples of a lattice
// stored row by row came from a few columns.  Tree build of 128 x 32 x 32 bodies:
// 214 us with radix passes, 1,180 with those samples, 147 with these.)
__device__ __forceinline__ int64_t sample_at(int i, int64_t n, int ns) {
  uint32_t h = (uint32_t)i;
  h = (h ^ h >> 16) * 0x85ebca6bu;
  h = (h ^ h >> 13) * 0xc2b2ae35u;
  h ^= h >> 16;
  return i * n / ns + ((int64_t)(h >> 16) * (n / ns) >> 16);
}
// the splitters of `buckets` buckets; a short input is sorted here and now.
// The samples are gathered into (tk, tv), kBlockSortMax entries of scratch
__global__ void __launch_bounds__(1024) k_sort_sample(uint64_t *keys, int32_t *vals,
                                                      const int64_t *d_n, int buckets, int kb,
                                                      int vb, SortWork *w, uint64_t *tk,
                                                      int32_t *tv) {
  pdl_wait();
  extern __shared__ __align__(16) unsigned char sort_mem[];
  uint64_t *sk = reinterpret_cast<uint64_t *>(sort_mem);
  int32_t *sv = reinterpret_cast<int32_t *>(sk + kBlockSortMax + kBlockSortMax / 8);
  const int64_t n = *d_n;
  const int t = threadIdx.x;
  const bool small = n <= kBlockSortMax;
  if (t < buckets) w->count[t] = 0;
  if (t == 0) w->done = small ? 1 : 0;
  if (small) {
    sort_entries(keys, vals, keys, vals, (int)n, 0, kb, vb, sk, sv);
    return;
  }
  const int per = kSamples / buckets < 8 ? kSamples / buckets : 8, ns = per * buckets;
  uint64_t k[kSamples / 1024];
  int32_t v[kSamples / 1024];
#pragma unroll
  for (int q = 0; q < kSamples / 1024; ++q) {
    const int i = t + q * 1024;
    const int64_t e = sample_at(i < ns ? i : 0, n, ns);
    k[q] = keys[e];
    v[q] = vals[e];
  }
#pragma unroll
  for (int q = 0; q < kSamples / 1024; ++q)
    if (t + q * 1024 < ns) { tk[t + q * 1024] = k[q]; tv[t + q * 1024] = v[q]; }
  __syncthreads();
  sort_entries(tk, tv, nullptr, nullptr, ns, 0, kb, vb, sk, sv);
  if (t > 0 && t < buckets) {
    w->skey[t - 1] = sk[slot(per * t)];
    w->sval[t - 1] = sv[slot(per * t)];
  }
}

constexpr int kClassThreads = 512;
constexpr int kClassPer = 4;
constexpr int kClassTile = kClassThreads * kClassPer;

// each key's bucket (the number of splitters at or below it, a power of two of
// buckets searched without branches) and its place in the bucket
__global__ void __launch_bounds__(kClassThreads) k_sort_class(const uint64_t *keys,
                                                              const int32_t *vals,
                                                              const int64_t *d_n, int buckets,
                                                              int kb, SortWork *w,
                                                              uint32_t *where) {
  pdl_wait();
  // searched by the splitters' leading 32 bits (half the shared-memory
  // conflicts of 64-bit words), the rest read on equality
  __shared__ uint32_t sl[kMaxBuckets];
  __shared__ uint64_t sk[kMaxBuckets];
  __shared__ int32_t sv[kMaxBuckets];
  __shared__ uint32_t h[kMaxBuckets];
  const int64_t n = *d_n, base = (int64_t)blockIdx.x * kClassTile;
  const int sh = kb > 32 ? kb - 32 : 0;
  const int t = threadIdx.x;
  if (base >= n || w->done) return;
  uint64_t k[kClassPer];
  int32_t v[kClassPer];
#pragma unroll
  for (int q = 0; q < kClassPer; ++q) {
    const int64_t e = base + q * kClassThreads + t;
    k[q] = e < n ? keys[e] : 0ull;
    v[q] = e < n ? vals[e] : 0;
  }
  for (int b = t; b < buckets; b += kClassThreads) {
    sk[b] = w->skey[b];
    sv[b] = w->sval[b];
    sl[b] = (uint32_t)(sk[b] >> sh);
    h[b] = 0;
  }
  __syncthreads();
  uint32_t bk[kClassPer] = {}, r[kClassPer];
  for (int step = buckets >> 1; step > 0; step >>= 1)
#pragma unroll
    for (int q = 0; q < kClassPer; ++q) {
      const int m = (int)bk[q] + step - 1;
      const uint32_t x = sl[m], kl = (uint32_t)(k[q] >> sh);
      if (x < kl || (x == kl && !pair_less(k[q], v[q], sk[m], sv[m]))) bk[q] += step;
    }
#pragma unroll
  for (int q = 0; q < kClassPer; ++q)
    r[q] = base + q * kClassThreads + t < n ? atomicAdd(&h[bk[q]], 1u) : 0u;
  __syncthreads();
  for (int b = t; b < buckets; b += kClassThreads)
    if (h[b]) h[b] = atomicAdd(&w->count[b], h[b]);
  __syncthreads();
#pragma unroll
  for (int q = 0; q < kClassPer; ++q) {
    const int64_t e = base + q * kClassThreads + t;
    if (e < n) where[e] = bk[q] << kPosBits | (h[bk[q]] + r[q]);
  }
}

__global__ void __launch_bounds__(kClassThreads) k_sort_move(const uint64_t *keys,
                                                             const int32_t *vals, uint64_t *okeys,
                                                             int32_t *ovals, const int64_t *d_n,
                                                             int buckets, SortWork *w,
                                                             const uint32_t *where) {
  pdl_wait();
  __shared__ int64_t sh[33];
  __shared__ uint32_t start[kMaxBuckets];
  const int64_t n = *d_n, base = (int64_t)blockIdx.x * kClassTile;
  const int t = threadIdx.x;
  if (base >= n || w->done) return;
  uint64_t k[kClassPer];
  int32_t v[kClassPer];
  uint32_t p[kClassPer];
#pragma unroll
  for (int q = 0; q < kClassPer; ++q) {
    const int64_t e = base + q * kClassThreads + t;
    if (e < n) { k[q] = keys[e]; v[q] = vals[e]; p[q] = where[e]; }
  }
  const uint32_t c0 = 2 * t < buckets ? w->count[2 * t] : 0u,
                 c1 = 2 * t + 1 < buckets ? w->count[2 * t + 1] : 0u;
  int64_t ex;
  block_excl_scan((int64_t)c0 + c1, &ex, sh);
  if (2 * t < kMaxBuckets) {
    start[2 * t] = (uint32_t)ex;
    start[2 * t + 1] = (uint32_t)ex + c0;
  }
  __syncthreads();
  if (blockIdx.x == 0) {
    for (int b = t; b < buckets; b += kClassThreads) w->start[b] = start[b];
    if (t == 0) w->start[buckets] = (uint32_t)n;
  }
#pragma unroll
  for (int q = 0; q < kClassPer; ++q)
    if (base + q * kClassThreads + t < n) {
      const uint32_t d = start[p[q] >> kPosBits] + (p[q] & ((1u << kPosBits) - 1u));
      okeys[d] = k[q];
      ovals[d] = v[q];
    }
}

// merges runs of r of the n entries of (ik, iv) into runs of 2 r of (ok, ov);
// thread t of nt takes the outputs from kItems t on
__device__ void merge_round(const uint64_t *ik, const int32_t *iv, uint64_t *ok, int32_t *ov, int n,
                            int r, int t, int nt) {
  for (int o = t * kItems; o < n; o += nt * kItems) {
    // a thread's outputs may cross into the next pair of runs
    int base = -1, ia = 0, ib = 0, a1 = 0, b1 = 0;
    for (int q = 0; q < kItems && o + q < n; ++q) {
      const int nb = (o + q) / (2 * r) * (2 * r);
      if (nb != base) {
        base = nb;
        const int diag = o + q - base;
        a1 = min(base + r, n);
        b1 = min(base + 2 * r, n);
        int lo = max(0, diag - (b1 - a1)), hi = min(diag, a1 - base);
        while (lo < hi) {
          const int mid = (lo + hi) >> 1, pa = base + mid, pb = a1 + diag - 1 - mid;
          if (pair_less(ik[pa], iv[pa], ik[pb], iv[pb])) lo = mid + 1; else hi = mid;
        }
        ia = base + lo;
        ib = a1 + diag - lo;
      }
      const bool ta = ib >= b1 || (ia < a1 && pair_less(ik[ia], iv[ia], ik[ib], iv[ib]));
      const int f = ta ? ia++ : ib++;
      ok[o + q] = ik[f];
      ov[o + q] = iv[f];
    }
  }
}

// a bucket a block, from (ik, iv) into (ok, ov); one that does not fit (rare)
// is sorted in runs that do, the runs then merged through global memory
__global__ void __launch_bounds__(kLocalThreads, 3) k_sort_local(uint64_t *ik, int32_t *iv,
                                                              uint64_t *ok, int32_t *ov,
                                                              int buckets, int key_bits, int vb,
                                                              const SortWork *w) {
  pdl_wait();
  extern __shared__ __align__(16) unsigned char sort_mem[];
  uint64_t *sk = reinterpret_cast<uint64_t *>(sort_mem);
  int32_t *sv = reinterpret_cast<int32_t *>(sk + kLocalMax + kLocalMax / 8);
  if (w->done) return;
  const int b = blockIdx.x;
  const uint32_t s0 = w->start[b];
  const int n = (int)(w->start[b + 1] - s0);
  // the bucket's keys lie between its splitters
  const uint64_t lo = b > 0 ? w->skey[b - 1] : 0ull;
  const uint64_t hi = b < buckets - 1 ? w->skey[b]
                                      : (key_bits < 64 ? (1ull << key_bits) - 1 : ~0ull);
  const int kb = 64 - __clzll((long long)(hi - lo));
  ik += s0; iv += s0; ok += s0; ov += s0;
  for (int c = 0; c < n; c += kLocalMax)
    sort_entries(ik + c, iv + c, ok + c, ov + c, min(kLocalMax, n - c), lo, kb, vb, sk, sv);
  for (int r = kLocalMax; r < n; r *= 2) {
    __threadfence_block();
    __syncthreads();
    // runs of r in (ok, ov) merged into (ik, iv), then copied back
    merge_round(ok, ov, ik, iv, n, r, threadIdx.x, kLocalThreads);
    __threadfence_block();
    __syncthreads();
    for (int i = threadIdx.x; i < n; i += kLocalThreads) { ok[i] = ik[i]; ov[i] = iv[i]; }
  }
}

// Entries of several systems, each segment's (at most P3T_SORT_SEGMENT) sorted
// by (key, value): one, two or four runs of equal length, a run a block, then
// merged pairwise.  The runs start in the buffer from which the merges end in
// (keys, vals).
__device__ __forceinline__ int segment_runs(int n) {
  return n <= kLocalMax ? 1 : (n <= 2 * kLocalMax ? 2 : 4);
}
__global__ void __launch_bounds__(kLocalThreads, 3) k_sort_runs(SegView seg, uint64_t *keys,
                                                             int32_t *vals, uint64_t *tk,
                                                             int32_t *tv, int kb, int vb) {
  pdl_wait();
  extern __shared__ __align__(16) unsigned char sort_mem[];
  uint64_t *sk = reinterpret_cast<uint64_t *>(sort_mem);
  int32_t *sv = reinterpret_cast<int32_t *>(sk + kLocalMax + kLocalMax / 8);
  const int d = blockIdx.x >> 2, q = blockIdx.x & 3;
  const int64_t s0 = seg_lo(seg, d);
  const int n = (int)(seg_hi(seg, d) - s0), runs = segment_runs(n);
  if (q >= runs) return;
  const int r = (n + runs - 1) / runs, n0 = q * r, len = min(r, n - n0);
  const int64_t o = s0 + n0;
  sort_entries(keys + o, vals + o, (runs == 2 ? tk : keys) + o, (runs == 2 ? tv : vals) + o, len, 0,
               kb, vb, sk, sv);
}
// the first merges of four runs (keys -> tk), or the last ones (tk -> keys)
constexpr int kMergeThreads = 256, kMergeBlocks = P3T_SORT_SEGMENT / (kMergeThreads * kItems);
__global__ void __launch_bounds__(kMergeThreads) k_merge_runs(SegView seg, uint64_t *keys,
                                                              int32_t *vals, uint64_t *tk,
                                                              int32_t *tv, bool last) {
  pdl_wait();
  const int d = blockIdx.x / kMergeBlocks, q = blockIdx.x % kMergeBlocks;
  const int64_t s0 = seg_lo(seg, d);
  const int n = (int)(seg_hi(seg, d) - s0), runs = segment_runs(n);
  if (runs < (last ? 2 : 4)) return;
  const int r = (n + runs - 1) / runs, t = q * kMergeThreads + threadIdx.x;
  constexpr int nt = kMergeBlocks * kMergeThreads;
  if (last)
    merge_round(tk + s0, tv + s0, keys + s0, vals + s0, n, runs == 4 ? 2 * r : r, t, nt);
  else
    merge_round(keys + s0, vals + s0, tk + s0, tv + s0, n, r, t, nt);
}

}  // namespace

int64_t p3t_scan_state_words(int64_t n_cap) {
  return 2 + (n_cap + kScanTile - 1) / kScanTile;
}

int p3t_scan_i32_to_i64(const int32_t *in, int64_t *out, const int64_t *d_n,
                        int64_t n_cap, int64_t *d_total, unsigned long long *state,
                        int64_t state_words, DevStatus *st, int64_t poll_limit,
                        cudaStream_t s) {
  int64_t G = (n_cap + kScanTile - 1) / kScanTile;
  if (G < 1) G = 1;
  if (G + 2 > state_words) return P3T_ERR_CAPACITY;
  pdl_launch(scan_onepass<false>, dim3((unsigned)G), dim3(kScanThreads), 0, s, in, out, d_n, d_total,
             state, st, poll_limit);
  p3t_note_launches(1);
  return cudaGetLastError() == cudaSuccess ? P3T_OK : P3T_ERR_CUDA;
}

int p3t_scan_flag_pairs(const int32_t *in, int64_t *out, const int64_t *d_n, int64_t n_cap,
                        int64_t *d_total, unsigned long long *state, int64_t state_words,
                        DevStatus *st, int64_t poll_limit, cudaStream_t s) {
  int64_t G = (n_cap + kScanTile - 1) / kScanTile;
  if (G < 1) G = 1;
  if (G + 2 > state_words) return P3T_ERR_CAPACITY;
  pdl_launch(scan_onepass<true>, dim3((unsigned)G), dim3(kScanThreads), 0, s, in, out, d_n, d_total,
             state, st, poll_limit);
  p3t_note_launches(1);
  return cudaGetLastError() == cudaSuccess ? P3T_OK : P3T_ERR_CUDA;
}

int64_t p3t_radix_hist_entries(int64_t n_cap) {
  int64_t ntiles = (n_cap + kSortTile - 1) / kSortTile;
  if (ntiles < 1) ntiles = 1;
  return ntiles * kRadix + kRadix;  // + the digit totals
}

int p3t_radix_sort(uint64_t **keys, int32_t **vals, uint64_t **keys_alt,
                   int32_t **vals_alt, const int64_t *d_n, int64_t n_cap,
                   int begin_bit, int end_bit, uint32_t *hist,
                   int64_t hist_cap, cudaStream_t s, int32_t *inv) {
  int64_t ntiles = (n_cap + kSortTile - 1) / kSortTile;
  if (ntiles < 1) ntiles = 1;
  if (ntiles * kRadix + kRadix > hist_cap) return P3T_ERR_CAPACITY;
  uint32_t *digit_total = hist + ntiles * kRadix;
  for (int shift = begin_bit; shift < end_bit; shift += kRadixBits) {
    pdl_launch(radix_upsweep, dim3((unsigned)ntiles), dim3(kSortThreads), 0, s, *keys, d_n, shift,
                                                            hist, (int)ntiles);
    pdl_launch(radix_row_scan, dim3(kRadix), dim3(kRadix), 0, s, hist, (int)ntiles, digit_total, d_n);
    pdl_launch(radix_downsweep, dim3((unsigned)ntiles), dim3(kSortThreads), 0, s, 
        *keys, *vals, *keys_alt, *vals_alt, d_n, shift, hist, (int)ntiles, digit_total,
        shift + kRadixBits >= end_bit ? inv : (int32_t *)nullptr);
    p3t_note_launches(3);
    uint64_t *tk = *keys; *keys = *keys_alt; *keys_alt = tk;
    int32_t *tv = *vals; *vals = *vals_alt; *vals_alt = tv;
  }
  return cudaGetLastError() == cudaSuccess ? P3T_OK : P3T_ERR_CUDA;
}

size_t p3t_sort_work_bytes() { return sizeof(SortWork); }

// dynamic shared memory above 48 KB is granted per function and device
static bool sort_attr(const void *f, size_t bytes) {
  return cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes) ==
         cudaSuccess;
}

bool p3t_sort_prepare() {
  return sort_attr((const void *)k_sort_block, sort_smem(kBlockSortMax)) &&
         sort_attr((const void *)k_sort_sample, sort_smem(kBlockSortMax)) &&
         sort_attr((const void *)k_sort_runs, sort_smem(kLocalMax)) &&
         sort_attr((const void *)k_sort_local, sort_smem(kLocalMax));
}

int p3t_sort_pairs(uint64_t **keys, int32_t **vals, uint64_t **keys_alt, int32_t **vals_alt,
                   const int64_t *d_n, int64_t n_cap, int key_bits, uint32_t *hist,
                   int64_t hist_cap, void *work, uint32_t *where, cudaStream_t s) {
  int vb = 1;  // bits of a value below n_cap
  while (vb < 31 && ((int64_t)1 << vb) < n_cap) ++vb;
  if (n_cap <= kBlockSortMax) {
    pdl_launch(k_sort_block, dim3(1), dim3(1024), sort_smem(kBlockSortMax), s, *keys, *vals, d_n,
               key_bits, vb);
    p3t_note_launches(1);
    return cudaGetLastError() == cudaSuccess ? P3T_OK : P3T_ERR_CUDA;
  }
  // four radix passes take less than the sample sort's launches
  if (n_cap > kSampleMax || key_bits <= 32)
    return p3t_radix_sort(keys, vals, keys_alt, vals_alt, d_n, n_cap, 0, key_bits, hist, hist_cap,
                          s);
  int buckets = 16;  // about 1,000 keys each
  while (buckets < kMaxBuckets && (int64_t)buckets * 1000 < n_cap) buckets *= 2;
  SortWork *w = static_cast<SortWork *>(work);
  const unsigned tiles = (unsigned)((n_cap + kClassTile - 1) / kClassTile);
  // the samples stand in the second buffers (n_cap > kBlockSortMax entries)
  // until the keys move there
  pdl_launch(k_sort_sample, dim3(1), dim3(1024), sort_smem(kBlockSortMax), s, *keys, *vals, d_n,
             buckets, key_bits, vb, w, *keys_alt, *vals_alt);
  pdl_launch(k_sort_class, dim3(tiles), dim3(kClassThreads), 0, s, *keys, *vals, d_n, buckets,
             key_bits, w, where);
  pdl_launch(k_sort_move, dim3(tiles), dim3(kClassThreads), 0, s, *keys, *vals, *keys_alt,
             *vals_alt, d_n, buckets, w, where);
  pdl_launch(k_sort_local, dim3((unsigned)buckets), dim3(kLocalThreads), sort_smem(kLocalMax), s,
             *keys_alt, *vals_alt, *keys, *vals, buckets, key_bits, vb, w);
  p3t_note_launches(4);
  return cudaGetLastError() == cudaSuccess ? P3T_OK : P3T_ERR_CUDA;
}

int p3t_sort_segments(const SegView &sv, uint64_t *keys, int32_t *vals, uint64_t *keys_alt,
                      int32_t *vals_alt, int64_t seg_max, int64_t n_cap, int key_bits, cudaStream_t s) {
  int vb = 1;  // bits of a value below n_cap
  while (vb < 31 && ((int64_t)1 << vb) < n_cap) ++vb;
  pdl_launch(k_sort_runs, dim3((unsigned)sv.nseg * 4), dim3(kLocalThreads), sort_smem(kLocalMax), s,
             sv, keys, vals, keys_alt, vals_alt, key_bits, vb);
  for (int last = seg_max > 2 * kLocalMax ? 0 : 1; last < 2 && seg_max > kLocalMax; ++last) {
    pdl_launch(k_merge_runs, dim3((unsigned)sv.nseg * kMergeBlocks), dim3(kMergeThreads), 0, s, sv,
               keys, vals, keys_alt, vals_alt, last == 1);
    p3t_note_launches(1);
  }
  p3t_note_launches(1);
  return cudaGetLastError() == cudaSuccess ? P3T_OK : P3T_ERR_CUDA;
}
