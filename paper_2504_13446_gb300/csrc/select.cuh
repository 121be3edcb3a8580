// select.cuh -- block-wide selection and sorting helpers (one CTA per query).
#pragma once

#include "common.cuh"

namespace rkr {

// Digit of an 8-bit histogram (by the calling warp, all lanes): the first bin whose
// running count reaches k, the keys below it subtracted from k.  Eight bins a lane,
// a scan over the lanes, then the lane's bins.
__device__ __forceinline__ void warp_digit(const uint32_t *hist, uint64_t k, int shift,
                                           uint64_t prefix, uint64_t *bc) {
  const int lane = threadIdx.x & 31;
  uint32_t h[8], sum = 0;
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    h[j] = hist[8 * lane + j];
    sum += h[j];
  }
  uint64_t incl = sum;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint64_t t = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += t;
  }
  const unsigned reach = __ballot_sync(0xffffffffu, incl >= k);
  // (the k-th smallest exists, so some lane reaches k)
  if (lane == (reach ? __ffs(reach) - 1 : 31)) {
    uint64_t acc = incl - sum;
    int sel = 7;
#pragma unroll
    for (int j = 7; j >= 0; --j) {   // the first bin whose running count reaches k
      uint64_t before = acc;
#pragma unroll
      for (int i = 0; i < j; ++i) before += h[i];
      if (before + h[j] >= k) sel = j;
    }
#pragma unroll
    for (int i = 0; i < 8; ++i)
      if (i < sel) acc += h[i];
    bc[0] = prefix | ((uint64_t)(8 * lane + sel) << shift);
    bc[1] = k - acc;
  }
}

// k-th smallest (1-based k) of the keys fn(i, key) yields for i in [0, cnt)
// (fn returns false for elements that do not take part).  MSB-first radix
// select on 8-bit digits over an nbits-wide key.  Every thread of the block must
// call it with the same arguments; the k-th smallest must exist.
// A thread evaluates four keys before it adds any to the histogram, so that
// their loads are in flight together: one CTA may have to walk a million keys.
template <class F>
__device__ uint64_t block_kth(int64_t cnt, uint64_t k, int nbits, F fn, uint32_t *hist,
                              uint64_t *bc) {
  uint64_t prefix = 0, mask = 0;
  const int64_t T = blockDim.x;
  for (int shift = nbits - 8; shift >= 0; shift -= 8) {
    for (int i = threadIdx.x; i < 256; i += blockDim.x) hist[i] = 0;
    __syncthreads();
    int64_t i = threadIdx.x;
    for (; i + 3 * T < cnt; i += 4 * T) {
      uint64_t key[4];
      bool in[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) in[j] = fn(i + j * T, key[j]);
#pragma unroll
      for (int j = 0; j < 4; ++j)
        if (in[j] && (key[j] & mask) == prefix) atomicAdd(&hist[(key[j] >> shift) & 255u], 1u);
    }
    for (; i < cnt; i += T) {
      uint64_t key;
      if (fn(i, key) && (key & mask) == prefix) atomicAdd(&hist[(key >> shift) & 255u], 1u);
    }
    __syncthreads();
    if (threadIdx.x < 32) warp_digit(hist, k, shift, prefix, bc);
    __syncthreads();
    prefix = bc[0];
    k = bc[1];
    mask |= (uint64_t)255 << shift;
    __syncthreads();
  }
  return prefix;
}

// The k-th smallest of two arrays of 32-bit keys (at most nbits wide) in the same
// passes; hist holds 512 bins, bc four words.  At least 64 threads.
__device__ __forceinline__ void block_kth_pair(const uint32_t *a, const uint32_t *b, int64_t cnt,
                                               uint64_t k, int nbits, uint32_t *hist, uint64_t *bc,
                                               uint64_t &ra, uint64_t &rb) {
  uint32_t pa = 0, pb = 0, mask = 0;
  uint64_t ka = k, kb = k;
  const int64_t T = blockDim.x;
  for (int shift = nbits - 8; shift >= 0; shift -= 8) {
    for (int i = threadIdx.x; i < 512; i += blockDim.x) hist[i] = 0;
    __syncthreads();
    int64_t i = threadIdx.x;
    auto add = [&](uint32_t x, uint32_t y) {
      if ((x & mask) == pa) atomicAdd(&hist[(x >> shift) & 255u], 1u);
      if ((y & mask) == pb) atomicAdd(&hist[256 + ((y >> shift) & 255u)], 1u);
    };
    for (; i + 3 * T < cnt; i += 4 * T) {
      uint32_t x[4], y[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        x[j] = a[i + j * T];
        y[j] = b[i + j * T];
      }
#pragma unroll
      for (int j = 0; j < 4; ++j) add(x[j], y[j]);
    }
    for (; i < cnt; i += T) add(a[i], b[i]);
    __syncthreads();
    if (threadIdx.x < 32) warp_digit(hist, ka, shift, pa, bc);
    else if (threadIdx.x < 64) warp_digit(hist + 256, kb, shift, pb, bc + 2);
    __syncthreads();
    pa = (uint32_t)bc[0];
    ka = bc[1];
    pb = (uint32_t)bc[2];
    kb = bc[3];
    mask |= 255u << shift;
    __syncthreads();
  }
  ra = pa;
  rb = pb;
}

// Number of i in [0, cnt) with pred(i).
template <class F>
__device__ int64_t block_count(int64_t cnt, F pred, unsigned long long *acc) {
  if (threadIdx.x == 0) *acc = 0;
  __syncthreads();
  unsigned long long mine = 0;
  for (int64_t i = threadIdx.x; i < cnt; i += blockDim.x) mine += pred(i) ? 1 : 0;
  for (int o = 16; o > 0; o >>= 1) mine += __shfl_xor_sync(0xffffffffu, mine, o);
  if ((threadIdx.x & 31) == 0 && mine) atomicAdd(acc, mine);
  __syncthreads();
  int64_t r = (int64_t)*acc;
  __syncthreads();
  return r;
}

// Entries sorted in shared memory: ascending by (k1, k2).
struct SortEnt {
  uint64_t k1;
  uint32_t k2;
  int32_t idx;
};

__device__ __forceinline__ bool ent_less(const SortEnt &a, const SortEnt &b) {
  return a.k1 < b.k1 || (a.k1 == b.k1 && a.k2 < b.k2);
}

// Bitonic sort of e[0 .. count) in shared memory; e must have room for the next
// power of two, the tail is padded with maximal keys.
__device__ void block_sort(SortEnt *e, int count) {
  int np2 = 1;
  while (np2 < count) np2 <<= 1;
  for (int i = count + threadIdx.x; i < np2; i += blockDim.x) {
    e[i].k1 = ~0ull;
    e[i].k2 = 0xffffffffu;
    e[i].idx = -1;
  }
  __syncthreads();
  // pair p of a step: i has bit j clear, its partner is i + j
  auto step = [&](int p, int k, int j) {
    const int i = ((p & ~(j - 1)) << 1) | (p & (j - 1));
    const bool asc = (i & k) == 0;
    const SortEnt a = e[i], b = e[i + j];
    if (ent_less(b, a) == asc) { e[i] = b; e[i + j] = a; }
  };
  if (np2 <= 64) {   // one warp, no block barriers
    if (threadIdx.x < 32)
      for (int k = 2; k <= np2; k <<= 1)
        for (int j = k >> 1; j > 0; j >>= 1) {
          if ((int)threadIdx.x < np2 / 2) step(threadIdx.x, k, j);
          __syncwarp();
        }
    __syncthreads();
    return;
  }
  for (int k = 2; k <= np2; k <<= 1)
    for (int j = k >> 1; j > 0; j >>= 1) {
      for (int p = threadIdx.x; p < np2 / 2; p += blockDim.x) step(p, k, j);
      __syncthreads();
    }
}

}  // namespace rkr
