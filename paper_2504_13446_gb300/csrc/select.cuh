// select.cuh -- block-wide selection and sorting helpers (one CTA per query).
#pragma once

#include "common.cuh"

namespace rkr {

// Digit of an 8-bit histogram (by the calling warp, all lanes): the first bin whose
// running count reaches k, the keys below it subtracted from k, the bin's count in
// *bin.  Eight bins a lane, a scan over the lanes, then the lane's bins.
__device__ __forceinline__ void warp_digit(const uint32_t *hist, uint32_t k, int shift,
                                           uint64_t prefix, uint64_t *bc, uint32_t *bin) {
  const int lane = threadIdx.x & 31;
  uint32_t h[8], sum = 0;
  const uint4 ha = reinterpret_cast<const uint4 *>(hist)[2 * lane];
  const uint4 hb = reinterpret_cast<const uint4 *>(hist)[2 * lane + 1];
  h[0] = ha.x; h[1] = ha.y; h[2] = ha.z; h[3] = ha.w;
  h[4] = hb.x; h[5] = hb.y; h[6] = hb.z; h[7] = hb.w;
#pragma unroll
  for (int j = 0; j < 8; ++j) sum += h[j];
  uint32_t incl = sum;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const uint32_t t = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += t;
  }
  const unsigned reach = __ballot_sync(0xffffffffu, incl >= k);
  // (the k-th smallest exists, so some lane reaches k)
  if (lane == (reach ? __ffs(reach) - 1 : 31)) {
    uint32_t before = incl - sum, acc = before;
    int sel = 0;
    uint32_t c = h[0];
#pragma unroll
    for (int j = 0; j < 7; ++j) {   // past every bin whose running count stays below k
      before += h[j];
      if (before < k) {
        sel = j + 1;
        acc = before;
        c = h[j + 1];
      }
    }
    bc[0] = prefix | ((uint64_t)(8 * lane + sel) << shift);
    bc[1] = k - acc;
    *bin = c;
  }
}

// k-th smallest (1-based k) of the keys fn(i, key) yields for i in [0, cnt)
// (fn returns false for elements that do not take part).  MSB-first radix
// select on 8-bit digits over an nbits-wide key.  Every thread of the block must
// call it with the same arguments; the k-th smallest must exist.
// A thread evaluates AHEAD keys before it adds any to the histogram, so that
// their loads are in flight together: one CTA may have to walk a million keys.
//
// The search ends early once at most `limit` keys lie at or below the bin that holds
// the k-th: their number is left in total and the bin's last key is returned (so
// limit 0 searches for the k-th itself).
template <int AHEAD = 4, class F>
__device__ uint64_t block_kth_cut(int64_t cnt, uint64_t k, int nbits, F fn, uint32_t *hist,
                                  uint64_t *bc, uint32_t limit, uint32_t &total) {
  uint64_t prefix = 0, mask = 0;
  uint32_t left = (uint32_t)k, bin = 0;
  __shared__ uint32_t bin_s;
  const int64_t T = blockDim.x;
  for (int i = threadIdx.x; i < 256; i += blockDim.x) hist[i] = 0;
  __syncthreads();
  for (int shift = nbits - 8; shift >= 0; shift -= 8) {
    int64_t i = threadIdx.x;
    for (; i + (AHEAD - 1) * T < cnt; i += AHEAD * T) {
      uint64_t key[AHEAD];
      bool in[AHEAD];
#pragma unroll
      for (int j = 0; j < AHEAD; ++j) in[j] = fn(i + j * T, key[j]);
#pragma unroll
      for (int j = 0; j < AHEAD; ++j)
        if (in[j] && (key[j] & mask) == prefix) atomicAdd(&hist[(key[j] >> shift) & 255u], 1u);
    }
    for (; i < cnt; i += T) {
      uint64_t key;
      if (fn(i, key) && (key & mask) == prefix) atomicAdd(&hist[(key >> shift) & 255u], 1u);
    }
    __syncthreads();
    if (threadIdx.x < 32) warp_digit(hist, left, shift, prefix, bc, &bin_s);
    __syncthreads();
    prefix = bc[0];
    left = (uint32_t)bc[1];
    bin = bin_s;
    mask |= (uint64_t)255 << shift;
    for (int z = threadIdx.x; z < 256; z += blockDim.x) hist[z] = 0;
    __syncthreads();
    if ((uint32_t)k - left + bin <= limit) break;
  }
  total = (uint32_t)k - left + bin;
  return (prefix | ~mask) & (~0ull >> (64 - nbits));
}

template <int AHEAD = 4, class F>
__device__ uint64_t block_kth(int64_t cnt, uint64_t k, int nbits, F fn, uint32_t *hist,
                              uint64_t *bc) {
  uint32_t total;
  return block_kth_cut<AHEAD>(cnt, k, nbits, fn, hist, bc, 0u, total);
}

// The k-th smallest of two arrays of 32-bit keys (at most nbits wide) in the same
// passes; hist holds 512 bins, bc four words.  At least 64 threads.  Up to four keys
// of each array a thread are loaded once and stay in registers over the passes.
__device__ __forceinline__ void block_kth_pair(const uint32_t *a, const uint32_t *b, int64_t cnt,
                                               uint64_t k, int nbits, uint32_t *hist, uint64_t *bc,
                                               uint64_t &ra, uint64_t &rb) {
  uint32_t pa = 0, pb = 0, mask = 0;
  uint32_t ka = (uint32_t)k, kb = (uint32_t)k;
  __shared__ uint32_t bin_s[2];
  const int64_t T = blockDim.x;
  const bool held = cnt <= 4 * T;
  uint32_t x[4], y[4];
  auto load = [&](int64_t i, int64_t end) {
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const bool in = i + j * T < end;
      x[j] = in ? a[i + j * T] : 0u;
      y[j] = in ? b[i + j * T] : 0u;
    }
  };
  if (held) load(threadIdx.x, cnt);
  for (int i = threadIdx.x; i < 512; i += blockDim.x) hist[i] = 0;
  __syncthreads();
  for (int shift = nbits - 8; shift >= 0; shift -= 8) {
    for (int64_t i = threadIdx.x; i < cnt; i += 4 * T) {
      if (!held) load(i, cnt);
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        if (i + j * T >= cnt) break;
        if ((x[j] & mask) == pa) atomicAdd(&hist[(x[j] >> shift) & 255u], 1u);
        if ((y[j] & mask) == pb) atomicAdd(&hist[256 + ((y[j] >> shift) & 255u)], 1u);
      }
    }
    __syncthreads();
    if (threadIdx.x < 32) warp_digit(hist, ka, shift, pa, bc, &bin_s[0]);
    else if (threadIdx.x < 64) warp_digit(hist + 256, kb, shift, pb, bc + 2, &bin_s[1]);
    __syncthreads();
    pa = (uint32_t)bc[0];
    ka = (uint32_t)bc[1];
    pb = (uint32_t)bc[2];
    kb = (uint32_t)bc[3];
    mask |= 255u << shift;
    for (int i = threadIdx.x; i < 512; i += blockDim.x) hist[i] = 0;
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

// Sort of e[0 .. count) in shared memory.  Few entries (count^2 <= 16 threads' worth,
// so 64 with 256 threads, 128 with 1,024): every entry's place is counted by 4 to 32
// threads (10 entries: 0.5 us; 21 bitonic steps in one warp 3 us).  More: bitonic; e
// must have room for the next power of two, the tail is padded with maximal keys.
__device__ void block_sort(SortEnt *e, int count) {
  __syncthreads();
  if (count * count <= 16 * (int)blockDim.x) {
    int per = 4;   // threads an entry
    while (per < 32 && 2 * per * count <= (int)blockDim.x) per <<= 1;
    const int i = threadIdx.x / per;
    SortEnt mine{0, 0, 0};
    int place = 0;
    if (i < count) {
      mine = e[i];
      for (int j = threadIdx.x & (per - 1); j < count; j += per) {
        const SortEnt o = e[j];
        place += ent_less(o, mine) || (j < i && !ent_less(mine, o));
      }
    }
    for (int o = per >> 1; o > 0; o >>= 1) place += __shfl_xor_sync(0xffffffffu, place, o);
    __syncthreads();
    if (i < count && (threadIdx.x & (per - 1)) == 0) e[place] = mine;
    __syncthreads();
    return;
  }
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
  for (int k = 2; k <= np2; k <<= 1)
    for (int j = k >> 1; j > 0; j >>= 1) {
      for (int p = threadIdx.x; p < np2 / 2; p += blockDim.x) step(p, k, j);
      __syncthreads();
    }
}

}  // namespace rkr
