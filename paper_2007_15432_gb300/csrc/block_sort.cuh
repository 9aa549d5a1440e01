// Sorts of distinct unsigned words in registers and shared memory: up to 256 by a
// warp, up to eight a thread by a block (primitives.cu: 64-bit key words,
// neighbours.cu: 32-bit members).
#pragma once

#include <stdint.h>

constexpr int kItems = 8;  // a thread's run of sorted words

// shared-memory slot of entry i (a word skipped every eight: a thread's runs
// start in different banks)
__device__ __forceinline__ int slot(int i) { return i + (i >> 3); }

template <typename T>
__device__ __forceinline__ void sort2(T &a, T &b) {
  const T x = a < b ? a : b;
  b = a < b ? b : a;
  a = x;
}

// the warp's 256 words, eight a lane in any order, into ascending order (lane l
// holds the places from 8 l on)
template <typename T>
__device__ __forceinline__ void warp_sort(T (&k)[kItems]) {
  const int lane = threadIdx.x & 31;
  // Batcher's odd-even merge sort of eight
#pragma unroll
  for (int p = 1; p < kItems; p <<= 1)
#pragma unroll
    for (int h = p; h > 0; h >>= 1)
#pragma unroll
      for (int j = h % p; j + h < kItems; j += 2 * h)
#pragma unroll
        for (int i = 0; i < h; ++i)
          if (j + i + h < kItems && (j + i) / (2 * p) == (j + i + h) / (2 * p))
            sort2(k[j + i], k[j + i + h]);
  // runs of L lanes -> runs of 2 L lanes: the second run taken backwards,
  // then half-cleaners across lanes and within the thread
#pragma unroll
  for (int L = 1; L < 32; L <<= 1) {
    T o[kItems];
#pragma unroll
    for (int q = 0; q < kItems; ++q)
      o[q] = __shfl_xor_sync(0xffffffffu, k[kItems - 1 - q], 2 * L - 1);
    const bool up = (lane & L) != 0;
#pragma unroll
    for (int q = 0; q < kItems; ++q) k[q] = (k[q] < o[q]) != up ? k[q] : o[q];
#pragma unroll
    for (int h = L >> 1; h > 0; h >>= 1) {
      const bool hi = (lane & h) != 0;
#pragma unroll
      for (int q = 0; q < kItems; ++q) {
        const T x = __shfl_xor_sync(0xffffffffu, k[q], h);
        k[q] = (k[q] < x) != hi ? k[q] : x;
      }
    }
#pragma unroll
    for (int h = kItems / 2; h > 0; h >>= 1)
#pragma unroll
      for (int q = 0; q < kItems; ++q)
        if (!(q & h)) sort2(k[q], k[q + h]);
  }
}

// the words [0, n) in shared memory sorted by the block: eight a thread by an
// odd-even merge network, up to 256 a warp by bitonic merges in registers
// (no barrier), then merge rounds through shared memory, each thread taking
// the eight outputs that its merge-path search gives it
template <typename T>
__device__ void sort_words(T *sk, int n) {
  const int i0 = threadIdx.x * kItems;
  const bool in = i0 < n;
  T k[kItems];
  if ((int)(threadIdx.x & ~31u) * kItems < n) {  // the warp holds entries
#pragma unroll
    for (int q = 0; q < kItems; ++q) k[q] = i0 + q < n ? sk[slot(i0 + q)] : (T)~(T)0;
    warp_sort(k);
#pragma unroll
    for (int q = 0; q < kItems; ++q)
      if (i0 + q < n) sk[slot(i0 + q)] = k[q];
  }
  __syncthreads();
  for (int w = 32 * kItems; w < n; w <<= 1) {
    if (in) {
      const int base = i0 & ~(2 * w - 1), diag = i0 - base;
      const int a1 = min(base + w, n), b1 = min(base + 2 * w, n);
      int lo = max(0, diag - (b1 - a1)), hi = min(diag, a1 - base);
      while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (sk[slot(base + mid)] < sk[slot(a1 + diag - 1 - mid)]) lo = mid + 1; else hi = mid;
      }
      int ia = base + lo, ib = a1 + diag - lo;
      T ka = ia < a1 ? sk[slot(ia)] : (T)~(T)0, kb = ib < b1 ? sk[slot(ib)] : (T)~(T)0;
#pragma unroll
      for (int q = 0; q < kItems; ++q) {
        const bool ta = ka <= kb;  // words are distinct but for the filler
        k[q] = ta ? ka : kb;
        ia += ta;
        ib += !ta;
        const int nx = ta ? ia : ib;
        const T nk = nx < (ta ? a1 : b1) ? sk[slot(nx)] : (T)~(T)0;
        if (ta) ka = nk; else kb = nk;
      }
    }
    __syncthreads();
    if (in) {
#pragma unroll
      for (int q = 0; q < kItems; ++q)
        if (i0 + q < n) sk[slot(i0 + q)] = k[q];
    }
    __syncthreads();
  }
}
