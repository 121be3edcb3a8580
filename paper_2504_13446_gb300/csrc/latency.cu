// latency.cu -- c-approximate queries one at a time (latency mode).
//
// The paper answers each query on its own: u.q for every user and the table
// lookup of Section 4.3 step 1 (its dominant cost, O(nd) per query), then the
// k-th smallest bounds, the Case A/B filter and the interpolation.  Per query
// this runs three launches with no host synchronization between them:
//
//   k_latency_scan     one pass over U (FP32, coalesced): u.q of every user by
//                      FP32 products with a rigorous error bound; the bin j of
//                      Section 4.3 step 1 from that interval (where it straddles
//                      a threshold, from a compensated product of the whole warp,
//                      and canonically only where that straddles one too);
//                      r_low, r_up numerators from the table; a histogram of the
//                      upper-bound numerators; the last CTA takes from it
//                      T >= R_up_k (the k-th smallest upper bound numerator), the
//                      bound of the users that can matter
//   k_latency_compact  the users with r_low <= T
//   k_select_approx    steps 1-3 on those users (query.cu)
//
// Every user that step 2 or 3 can return has r_low <= R_up_k (Case A takes the
// k smallest r_up, all <= R_up_k, and r_low <= r_up; Case B prunes r_low >
// R_up_k), and R_low_k <= R_up_k <= T, so the k smallest lower and upper
// bounds lie among the compacted users: the answer equals the batched one bit
// for bit.  The scan is bound by HBM: it reads U once (4d bytes per user) and
// a few bytes of per-user data and table cells.
#include <math.h>
#include <stddef.h>
#include <string.h>

#include <new>

#include "index.cuh"

namespace rkr {
namespace lat {

constexpr int kLatThreads = 256;
constexpr int kLatBins = 2048;

// Bound factor of the scan's products: a term passes at most (d + 31) / 32 * 4
// FMAs of its lane's chain and three (bulk form: one chain of eight, five)
// additions of the reduction, each rounding by at most 2^-24 of a partial sum,
// and every partial sum is at most sum_k |u_k q_k| <= ||u|| ||q||; the canonical
// FP64 sum differs from the exact value by at most d 2^-53 ||u|| ||q||.
__host__ __device__ inline float latency_cfac(int d) {
  const double c = ((double)((d + 31) / 32 * 4 + 8) * 0x1p-24 + (double)d * 0x1p-53 + 0x1p-40) *
                   (1.0 + 0x1p-20);
  return (float)c * (1.0f + 0x1p-20f);
}

// Arguments of the scan kernels.
struct ScanArgs {
  const float *U;
  int64_t n;
  int d;
  const float *q, *qn;          // query row and its norm bound
  const float *unrm;
  const BinFP *bf;
  const double *fmin, *delta;
  const uint32_t *N;
  int tau;
  uint32_t top;
  int shift;
  uint32_t *nlo, *nup;          // per user
  int32_t *jout;
  uint32_t *ghist;              // kLatBins, zero between launches
  unsigned int *done;           // CTAs that have added their histogram, 0 between launches
  const int32_t *kq;            // k of the query
  uint32_t *T, *qcount;         // cut, candidate count (zeroed for the compaction)
  unsigned long long *nfp64;
  uint32_t wait;                // rounds a consumer warp of the bulk form waits for a stage
  const uint32_t *wait_p;       // the same read on the device (a captured launch), or null
};

// Finish of the warp's users (every lane calls it; lane's user u if live, with its
// product dot and the bound factors): the bin of u.q, the table's bounds, the
// histogram.  A lane whose interval straddles a threshold has its row taken again
// by the whole warp as a compensated product: one lane's canonical product here
// would hold its SM's FP64 pipe for d dependent steps.
__device__ __forceinline__ void finish_users(const ScanArgs &a, const float *qs, float cf,
                                             float qn, int64_t u, bool live, float dot,
                                             uint32_t *hist, uint32_t &fp64) {
  const int lane = threadIdx.x & 31;
  int j = 0, jhi = 0;
  if (live) {
    const BinFP bu = a.bf[u];
    const float b = __fadd_ru(__fmul_ru(__fmul_ru(cf, a.unrm[u]), qn), 1e-30f);
    const float lo = __fsub_rd(dot, b), hi = __fadd_ru(dot, b);
    const TightBins tb(bu);
    if (tb.usable()) {
      j = tb.lo(lo, a.tau);
      jhi = tb.hi(hi, a.tau);
    } else {
      bin_interval(bu, a.fmin[u], a.tau, lo, hi, j, jhi);
    }
  }
  unsigned open = __ballot_sync(0xffffffffu, live && j != jhi);
  while (open) {
    const int src = __ffs(open) - 1;
    open &= open - 1;
    const int64_t us = __shfl_sync(0xffffffffu, u, src);
    const float *row = a.U + us * a.d;
    Dot2 t;
    for (int k = lane; k < a.d; k += 32) t.add(row[k], qs[k]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const float p2 = __shfl_xor_sync(0xffffffffu, t.p, o);
      const float s2 = __shfl_xor_sync(0xffffffffu, t.s, o);
      const float a2 = __shfl_xor_sync(0xffffffffu, t.asum, o);
      const float sum = __fadd_rn(t.p, p2);
      const float z = __fsub_rn(sum, t.p);
      const float e = __fadd_rn(__fsub_rn(t.p, __fsub_rn(sum, z)), __fsub_rn(p2, z));
      t.p = sum;
      t.s = __fadd_rn(t.s, __fadd_rn(s2, e));
      t.asum = __fadd_ru(t.asum, a2);
    }
    if (lane == src) {
      const double res = (double)t.p + (double)t.s, E = (double)t.err(a.d + 8);
      const double fm = a.fmin[u], dl = a.delta[u];
      const double tlo = res - E, thi = res + E;
      int jl = exact_j(tlo, fm, dl, a.tau);
      // (NaN ends, of products beyond the range of float, decide nothing)
      if (!(tlo <= thi) || jl != exact_j(thi, fm, dl, a.tau)) {
        ++fp64;
        jl = exact_j(canon_dot_slow(row, qs, a.d), fm, dl, a.tau);
      }
      j = jl;
    }
  }
  if (live) {
    const uint32_t lo = j < a.tau ? a.N[u * a.tau + j] : 0u;
    const uint32_t up = j >= 1 ? a.N[u * a.tau + j - 1] : a.top;
    a.nlo[u] = lo;
    a.nup[u] = up;
    a.jout[u] = j;
    // lanes with the same bin add once (upper bounds crowd into few bins)
    const unsigned bin = min(up >> a.shift, (uint32_t)(kLatBins - 1));
    const unsigned peers = __match_any_sync(__activemask(), bin);
    if (lane == __ffs(peers) - 1) atomicAdd(&hist[bin], (uint32_t)__popc(peers));
  }
}

// End of a scan CTA: its histogram is added to the query's (most bins are empty),
// and the last CTA to do so finds T = upper end of the bin holding the k-th
// smallest upper-bound numerator (so T >= R_up_k), zeroes the query's candidate
// count and leaves the histogram and the counter at zero for the next launch.  A scan
// that timed out may have counted fewer than k users: T is then 0.  Either way the
// compaction starts from a count of zero, so it stays within its n slots.
__device__ __forceinline__ void flush_and_cut(const ScanArgs &a, uint32_t *hist, uint32_t fp64) {
  __shared__ uint32_t wsum[8];
  __shared__ int is_last;
  fp64 = __reduce_add_sync(0xffffffffu, fp64);
  if ((threadIdx.x & 31) == 0 && fp64) atomicAdd(a.nfp64, (unsigned long long)fp64);
  __syncthreads();
  for (int i = threadIdx.x; i < kLatBins; i += blockDim.x)
    if (hist[i]) atomicAdd(&a.ghist[i], hist[i]);
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) is_last = atomicAdd(a.done, 1u) == gridDim.x - 1;
  __syncthreads();
  if (!is_last) return;
  __threadfence();
  constexpr int kPer = kLatBins / 256;
  const int t = threadIdx.x, lane = t & 31;
  uint32_t h[kPer], sum = 0, incl = 0;
  if (t < 256) {
#pragma unroll
    for (int i = 0; i < kPer; ++i) {
      h[i] = __ldcg(&a.ghist[kPer * t + i]);
      a.ghist[kPer * t + i] = 0;
      sum += h[i];
    }
    incl = sum;
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t x = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += x;
    }
    if (lane == 31) wsum[t >> 5] = incl;
  }
  if (t == 0) {
    *a.T = 0;
    *a.qcount = 0;
    *a.done = 0;
  }
  __syncthreads();
  if (t < 256) {
    for (int w = 0; w < (t >> 5); ++w) incl += wsum[w];
    const uint32_t k = (uint32_t)*a.kq;
    uint32_t run = incl - sum;
    if (run < k && incl >= k) {
      int bin = kPer * t;
#pragma unroll
      for (int i = 0; i < kPer; ++i) {
        if (run < k && run + h[i] >= k) bin = kPer * t + i;
        run += h[i];
      }
      const uint64_t hi = ((uint64_t)(bin + 1) << a.shift) - 1;
      *a.T = bin == kLatBins - 1 || hi > 0xffffffffull ? 0xffffffffu : (uint32_t)hi;
    }
  }
}

// One pass over U: a warp takes 32 rows per iteration, four at a time with eight
// lanes each (16-byte loads where VEC = 4: 128 contiguous bytes of a row per load
// and row; single floats otherwise), so that a product costs three shuffles for
// four rows, and lane l finishes one of the 32 users.  Bound by HBM: 4 d bytes per
// user and about 60 more of bounds, table cells and results.  1M users at d = 200:
// 159 us (5.0 TB/s of the rows alone); with two or four groups of rows in flight
// per warp 194 and 268 us.
template <int VEC>
__global__ void __launch_bounds__(kLatThreads, 4) k_latency_scan(const ScanArgs a) {
  __shared__ __align__(16) float qs[kMaxD];
  __shared__ __align__(16) uint32_t hist[kLatBins];
  for (int i = threadIdx.x; i < kMaxD; i += blockDim.x) qs[i] = i < a.d ? a.q[i] : 0.0f;
  for (int i = threadIdx.x; i < kLatBins; i += blockDim.x) hist[i] = 0;
  __syncthreads();
  const float qn = *a.qn;
  const float cf = latency_cfac(a.d);
  const int lane = threadIdx.x & 31, sub = lane & 7, grp = lane >> 3;
  const int64_t gw = (int64_t)blockIdx.x * (kLatThreads / 32) + (threadIdx.x >> 5);
  const int64_t nw = (int64_t)gridDim.x * (kLatThreads / 32);
  [[maybe_unused]] constexpr int kPieces = kMaxD / (8 * VEC);   // per lane and row, at most
  const int pieces = (a.d + 8 * VEC - 1) / (8 * VEC);
  uint32_t fp64 = 0;
  for (int64_t r0 = gw * 32; r0 < a.n; r0 += nw * 32) {
    float mine = 0.0f;
#pragma unroll 1
    for (int sb = 0; sb < 8; ++sb) {
      const int64_t row = r0 + sb * 4 + grp;
      const bool ok = row < a.n;
      float acc = 0.0f;
      if constexpr (VEC == 4) {
        const float4 *r4 = reinterpret_cast<const float4 *>(a.U + row * a.d);
        const float4 *q4 = reinterpret_cast<const float4 *>(qs);
        const int dv = a.d >> 2;
        float4 x[kPieces];
#pragma unroll
        for (int p = 0; p < kPieces; ++p) {
          const int c = sub + 8 * p;
          x[p] = p < pieces && ok && c < dv ? __ldcs(r4 + c) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
#pragma unroll
        for (int p = 0; p < kPieces; ++p) {
          if (p < pieces) {
            const float4 y = q4[sub + 8 * p];   // zero beyond d
            acc = __fmaf_rn(x[p].x, y.x, acc);
            acc = __fmaf_rn(x[p].y, y.y, acc);
            acc = __fmaf_rn(x[p].z, y.z, acc);
            acc = __fmaf_rn(x[p].w, y.w, acc);
          }
        }
      } else {
        const float *rp = a.U + row * a.d;
#pragma unroll 8
        for (int p = 0; p < pieces; ++p) {
          const int c = sub + 8 * p;
          if (ok && c < a.d) acc = __fmaf_rn(__ldg(rp + c), qs[c], acc);
        }
      }
#pragma unroll
      for (int o = 4; o > 0; o >>= 1)
        acc = __fadd_rn(acc, __shfl_xor_sync(0xffffffffu, acc, o));
      if (sub == sb) mine = acc;
    }
    const int64_t u = r0 + sub * 4 + grp;
    finish_users(a, qs, cf, qn, u, u < a.n, mine, hist, fp64);
  }
  flush_and_cut(a, hist, fp64);
}

// ------------------------------------------------------------------
// Bulk-staged form (d a multiple of 4): the rows of U are contiguous, so a chunk
// of kBulkRows users is one cp.async.bulk copy.  Warp kBulkWarps (one lane)
// streams chunks into a ring of kBulkStages shared-memory stages; warps
// 0..kBulkWarps-1 each take kBulkRows / kBulkWarps rows of a stage, free the
// stage as soon as their products are formed, then finish their users.  One CTA
// per SM; every wait is bounded.  A timeout sets *err; whichever side gave up, the
// producer waits for the copies it issued before the CTA ends.
constexpr int kBulkWarps = 8;
constexpr int kBulkRows = 64;
constexpr int kBulkStages = 3;
constexpr int kBulkRowsPerWarp = kBulkRows / kBulkWarps;   // 8
constexpr uint32_t kBulkWait = 1u << 22;

__device__ __forceinline__ uint32_t bulk_smem(const void *p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ bool bulk_wait(uint64_t *bar, uint32_t parity,
                                          uint32_t limit = kBulkWait) {
  const uint32_t addr = bulk_smem(bar);
  for (uint32_t i = 0; i < limit; ++i) {
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
        " selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(addr), "r"(parity)
        : "memory");
    if (ok) return true;
  }
  return false;
}

size_t bulk_smem_bytes(int d) {
  return 128 + (size_t)kBulkStages * kBulkRows * d * 4 + 16 * kBulkStages +
         sizeof(float) * kMaxD + sizeof(uint32_t) * kLatBins;
}

__global__ void __launch_bounds__((kBulkWarps + 1) * 32, 1)
    k_latency_scan_bulk(const ScanArgs a, int *__restrict__ err) {
  const float *U = a.U;
  const int64_t n = a.n;
  const int d = a.d;
  extern __shared__ __align__(128) unsigned char bsm[];
  unsigned char *base = (unsigned char *)(((uintptr_t)bsm + 127) & ~(uintptr_t)127);
  const size_t stage_bytes = (size_t)kBulkRows * d * 4;
  unsigned char *stages = base;
  uint64_t *full = (uint64_t *)(stages + kBulkStages * stage_bytes);
  uint64_t *empty = full + kBulkStages;
  float *qs = (float *)(empty + kBulkStages);
  uint32_t *hist = (uint32_t *)(qs + kMaxD);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int i = threadIdx.x; i < kMaxD; i += blockDim.x) qs[i] = i < d ? a.q[i] : 0.0f;
  for (int i = threadIdx.x; i < kLatBins; i += blockDim.x) hist[i] = 0;
  if (threadIdx.x == 0) {
    for (int s = 0; s < kBulkStages; ++s) {
      asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bulk_smem(&full[s])), "r"(1));
      asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bulk_smem(&empty[s])),
                   "r"(kBulkWarps));
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  const int64_t nch = (n + kBulkRows - 1) / kBulkRows;
  bool failed = false;
  uint32_t fp64 = 0;
  if (warp == kBulkWarps) {
    // ------------------------------------------------------------ producer
    if (lane == 0) {
      uint32_t it = 0;
      for (int64_t ch = blockIdx.x; ch < nch; ch += gridDim.x, ++it) {
        const int s = it % kBulkStages;
        if (!bulk_wait(&empty[s], ((it / kBulkStages) & 1) ^ 1)) { failed = true; break; }
        const int64_t rows = min((int64_t)kBulkRows, n - ch * kBulkRows);
        const uint32_t bytes = (uint32_t)(rows * d * 4);
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(
                         bulk_smem(&full[s])),
                     "r"(bytes)
                     : "memory");
        asm volatile(
            "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, "
            "[%3];" ::"r"(bulk_smem(stages + s * stage_bytes)),
            "l"(reinterpret_cast<uint64_t>(U + ch * kBulkRows * d)), "r"(bytes),
            "r"(bulk_smem(&full[s]))
            : "memory");
      }
      if (failed) atomicExch(err, 1);
      // the copies issued land before the CTA can exit (a consumer that gave up did
      // not wait for them)
      for (uint32_t j = (it > kBulkStages ? it - kBulkStages : 0); j < it; ++j)
        bulk_wait(&full[j % kBulkStages], (j / kBulkStages) & 1);
    }
  } else {
    // ------------------------------------------------------------ consumers
    const float qn = *a.qn;
    const uint32_t limit = a.wait_p ? *a.wait_p : a.wait;
    const float cf = latency_cfac(d);
    const float4 *q4 = reinterpret_cast<const float4 *>(qs);
    const float4 b0 = q4[lane], b1 = q4[lane + 32];
    const int dv = d >> 2;
    uint32_t it = 0;
    for (int64_t ch = blockIdx.x; ch < nch; ch += gridDim.x, ++it) {
      const int s = it % kBulkStages;
      // (one answer for the warp: its lanes meet in shuffles below)
      if (!__all_sync(0xffffffffu, bulk_wait(&full[s], (it / kBulkStages) & 1, limit))) {
        failed = true;
        break;
      }
      const float *st = (const float *)(stages + s * stage_bytes);
      const int64_t u0 = ch * kBulkRows + warp * kBulkRowsPerWarp;
      float mine = 0.0f;
#pragma unroll
      for (int rr = 0; rr < kBulkRowsPerWarp; ++rr) {
        const float4 *r4 =
            reinterpret_cast<const float4 *>(st + (size_t)(warp * kBulkRowsPerWarp + rr) * d);
        float acc = 0.0f;
        if (u0 + rr < n) {
          if (lane < dv) {
            const float4 x = r4[lane];
            acc = __fmaf_rn(x.x, b0.x, acc);
            acc = __fmaf_rn(x.y, b0.y, acc);
            acc = __fmaf_rn(x.z, b0.z, acc);
            acc = __fmaf_rn(x.w, b0.w, acc);
          }
          if (lane + 32 < dv) {
            const float4 x = r4[lane + 32];
            acc = __fmaf_rn(x.x, b1.x, acc);
            acc = __fmaf_rn(x.y, b1.y, acc);
            acc = __fmaf_rn(x.z, b1.z, acc);
            acc = __fmaf_rn(x.w, b1.w, acc);
          }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
          acc = __fadd_rn(acc, __shfl_xor_sync(0xffffffffu, acc, o));
        if (lane == rr) mine = acc;
      }
      // this warp is done with the stage
      __syncwarp();
      if (lane == 0)
        asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bulk_smem(&empty[s]))
                     : "memory");
      const int64_t u = u0 + lane;
      finish_users(a, qs, cf, qn, u, lane < kBulkRowsPerWarp && u < n, mine, hist, fp64);
    }
    if (failed && lane == 0) atomicExch(err, 2);
  }
  flush_and_cut(a, hist, fp64);
}

// Users with r_low <= T, four a thread (their lower bounds in one load), slots by
// one atomic per warp.
__global__ void k_latency_compact(int64_t n, const uint32_t *__restrict__ nlo,
                                  const uint32_t *__restrict__ nup, const int32_t *__restrict__ j,
                                  const uint32_t *__restrict__ T, int q,
                                  uint32_t *__restrict__ qcount, int32_t *__restrict__ cu,
                                  uint32_t *__restrict__ clo, uint32_t *__restrict__ cup,
                                  int32_t *__restrict__ cj, double *__restrict__ cth) {
  const uint32_t t = *T;
  const int lane = threadIdx.x & 31;
  const int64_t u0 = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) * 4;
  uint32_t lo[4];
  if (u0 + 3 < n) {   // nlo is 256-byte aligned
    const uint4 v = *reinterpret_cast<const uint4 *>(nlo + u0);
    lo[0] = v.x; lo[1] = v.y; lo[2] = v.z; lo[3] = v.w;
  } else {
    for (int e = 0; e < 4; ++e) lo[e] = u0 + e < n ? nlo[u0 + e] : 0u;
  }
  int mine = 0;
#pragma unroll
  for (int e = 0; e < 4; ++e) mine += u0 + e < n && lo[e] <= t;
  int incl = mine;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int x = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += x;
  }
  const int total = __shfl_sync(0xffffffffu, incl, 31);
  if (total == 0) return;
  uint32_t base = 0;
  if (lane == 0) base = atomicAdd(&qcount[q], (uint32_t)total);
  base = __shfl_sync(0xffffffffu, base, 0);
  uint32_t pos = base + (uint32_t)(incl - mine);
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    const int64_t u = u0 + e;
    if (u >= n || lo[e] > t) continue;
    cu[pos] = (int32_t)u;
    clo[pos] = lo[e];
    cup[pos] = nup[u];
    cj[pos] = j[u];
    cth[pos] = __longlong_as_double(0x7ff8000000000000ll);  // u.q formed on demand
    ++pos;
  }
}

// Step-3 estimate of each compacted candidate (canonical u.q) and its outputs at
// `base`, with global user ids (local id + user_offset).
__global__ void k_candidate_out(const uint32_t *__restrict__ qcount, int q,
                                const int32_t *__restrict__ cu, const uint32_t *__restrict__ clo,
                                const uint32_t *__restrict__ cup, const int32_t *__restrict__ cj,
                                const float *__restrict__ U, const float *__restrict__ qrow, int d,
                                const double *__restrict__ fmin, const double *__restrict__ delta,
                                int tau, uint32_t s, int64_t user_offset, int64_t base,
                                int32_t *__restrict__ ou, uint32_t *__restrict__ olo,
                                uint32_t *__restrict__ oup, double *__restrict__ oest) {
  const int64_t cnt = qcount[q];
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < cnt;
       i += (int64_t)gridDim.x * blockDim.x) {
    const int64_t u = cu[i];
    const double th = canon_dot(U + u * d, qrow, d);
    ou[base + i] = (int32_t)(u + user_offset);
    olo[base + i] = clo[i];
    oup[base + i] = cup[i];
    oest[base + i] = interp_est(th, cj[i], clo[i], cup[i], fmin[u], delta[u], tau, s);
  }
}

// Scratch of the per-query bounds pass.
struct ScanBufs {
  uint32_t *nlo, *nup, *ghist, *T, *qcount;   // ghist: kLatBins, then the CTA counter
  int32_t *jall;
  unsigned long long *nfp64;   // [0] canonical evaluations, [1] select error, [2] scan error
  int *err;                    // the scan's error word (nfp64[2] unless replaced)
  const uint32_t *wait_p;      // see ScanArgs
  int grid, shift;
  uint32_t top;
  bool vec4, bulk;
  size_t bulk_smem;
};

rkr_status alloc_scan(const rkr_index *idx, int nq, int ctas_per_sm, DevBuf (&b)[7], ScanBufs &sb,
                      cudaStream_t st) {
  const int64_t n = idx->n;
  sb.top = (uint32_t)(idx->m * idx->s);
  sb.shift = 0;
  while ((sb.top >> sb.shift) >= (uint32_t)kLatBins) ++sb.shift;
  sb.vec4 = (idx->d % 4) == 0 && ((uintptr_t)idx->U % 16) == 0;
  int occ = 0;
  if (sb.vec4)
    RKR_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_latency_scan<4>, kLatThreads, 0));
  else
    RKR_CUDA(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, k_latency_scan<1>, kLatThreads, 0));
  occ = std::max(occ, 1);
  if (ctas_per_sm > 0) occ = std::min(occ, ctas_per_sm);
  const int64_t warps_needed = (n + 31) / 32;
  sb.grid = (int)std::max<int64_t>(
      1, std::min<int64_t>((int64_t)sm_count() * occ,
                           (warps_needed + kLatThreads / 32 - 1) / (kLatThreads / 32)));
  // bulk-staged scan: rows of a multiple of 16 bytes and a U base aligned to 16
  sb.bulk = tuning().latency_bulk && sb.vec4;
  if (sb.bulk) {
    sb.bulk_smem = bulk_smem_bytes(idx->d);
    RKR_CUDA(cudaFuncSetAttribute(k_latency_scan_bulk,
                                  cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  (int)sb.bulk_smem));
    sb.grid = (int)std::max<int64_t>(
        1, std::min<int64_t>(sm_count(), (n + kBulkRows - 1) / kBulkRows));
  }
  RKR_TRY(tmp_alloc(b[0], &sb.nlo, n, st));
  RKR_TRY(tmp_alloc(b[1], &sb.nup, n, st));
  RKR_TRY(tmp_alloc(b[2], &sb.jall, n, st));
  RKR_TRY(tmp_alloc(b[3], &sb.ghist, kLatBins + 1, st));
  RKR_TRY(tmp_alloc(b[4], &sb.T, 1, st));
  RKR_TRY(tmp_alloc(b[5], &sb.qcount, nq, st));
  RKR_TRY(tmp_alloc(b[6], &sb.nfp64, 3, st));
  sb.err = (int *)(sb.nfp64 + 2);
  sb.wait_p = nullptr;
  RKR_CUDA(cudaMemsetAsync(sb.ghist, 0, sizeof(uint32_t) * (kLatBins + 1), st));
  RKR_CUDA(cudaMemsetAsync(sb.qcount, 0, sizeof(uint32_t) * nq, st));
  RKR_CUDA(cudaMemsetAsync(sb.nfp64, 0, 3 * sizeof(unsigned long long), st));
  return RKR_OK;
}

// Bounds of every user for query q, their histogram and the cut T.
rkr_status scan_pass(const rkr_index *idx, const QueryCommon &qc, int q, const ScanBufs &sb,
                     cudaStream_t st) {
  const float *qrow = qc.Qd + (int64_t)q * idx->d;
  {
    ProfScope prof("k_latency_scan", st,
                   (double)idx->n * (4.0 * idx->d + 4 + sizeof(BinFP) + 8 + 8 + 12));
    ScanArgs a;
    a.U = idx->U; a.n = idx->n; a.d = idx->d; a.q = qrow; a.qn = qc.qnrm + q;
    a.unrm = idx->unrm; a.bf = idx->binfp; a.fmin = idx->fmin; a.delta = idx->delta;
    a.N = idx->N; a.tau = idx->tau; a.top = sb.top; a.shift = sb.shift;
    a.nlo = sb.nlo; a.nup = sb.nup; a.jout = sb.jall;
    a.ghist = sb.ghist; a.done = sb.ghist + kLatBins; a.kq = qc.kq_d + q;
    a.T = sb.T; a.qcount = sb.qcount + q; a.nfp64 = sb.nfp64;
    a.wait = epi_wait_limit();
    a.wait_p = sb.wait_p;
    if (sb.bulk)
      k_latency_scan_bulk<<<sb.grid, (kBulkWarps + 1) * 32, sb.bulk_smem, st>>>(
          a, sb.err);
    else if (sb.vec4)
      k_latency_scan<4><<<sb.grid, kLatThreads, 0, st>>>(a);
    else
      k_latency_scan<1><<<sb.grid, kLatThreads, 0, st>>>(a);
    note_launch();
  }
  RKR_CUDA(cudaGetLastError());
  return RKR_OK;
}

}  // namespace lat

using namespace lat;

// Per query, the users of this index whose lower bound is at most an upper
// estimate T of this index's R_up_k, with their bounds and step-3 estimates.
rkr_status run_query_approx_candidates(const rkr_index *idx, const QueryCommon &qc, int nq,
                                       int64_t user_offset, int64_t capacity, int64_t *offs_host,
                                       int32_t *users_d, uint32_t *nlo_d, uint32_t *nup_d,
                                       double *est_d, cudaStream_t st) {
  const int64_t n = idx->n;
  const int d = idx->d;
  DevBuf bs[7], b7, b8, b9, b10, b11;
  ScanBufs sb;
  RKR_TRY(alloc_scan(idx, nq, tuning().latency_ctas_per_sm, bs, sb, st));
  uint32_t *clo, *cup;
  int32_t *cu, *cj;
  double *cth;
  RKR_TRY(tmp_alloc(b7, &cu, n, st));
  RKR_TRY(tmp_alloc(b8, &clo, n, st));
  RKR_TRY(tmp_alloc(b9, &cup, n, st));
  RKR_TRY(tmp_alloc(b10, &cj, n, st));
  RKR_TRY(tmp_alloc(b11, &cth, n, st));
  const unsigned cgrid = (unsigned)((n + 1023) / 1024);   // four users a thread
  offs_host[0] = 0;
  for (int q = 0; q < nq; ++q) {
    const float *qrow = qc.Qd + (int64_t)q * d;
    RKR_TRY(scan_pass(idx, qc, q, sb, st));
    k_latency_compact<<<cgrid, 256, 0, st>>>(n, sb.nlo, sb.nup, sb.jall, sb.T, q, sb.qcount, cu,
                                             clo, cup, cj, cth);
    note_launch();
    RKR_CUDA(cudaGetLastError());
    uint32_t cnt = 0;
    RKR_CUDA(cudaMemcpyAsync(&cnt, sb.qcount + q, sizeof(cnt), cudaMemcpyDeviceToHost, st));
    RKR_CUDA(cudaStreamSynchronize(st));
    offs_host[q + 1] = offs_host[q] + cnt;
    if (offs_host[q + 1] <= capacity && cnt > 0) {
      k_candidate_out<<<(unsigned)std::min<int64_t>((cnt + 255) / 256, 4 * sm_count()), 256, 0,
                        st>>>(sb.qcount, q, cu, clo, cup, cj, idx->U, qrow, d, idx->fmin,
                              idx->delta, idx->tau, (uint32_t)idx->s, user_offset, offs_host[q],
                              users_d, nlo_d, nup_d, est_d);
      note_launch();
      RKR_CUDA(cudaGetLastError());
    }
  }
  RKR_CUDA(cudaStreamSynchronize(st));
  {
    unsigned long long h[3] = {0, 0, 0};
    RKR_CUDA(cudaMemcpy(h, sb.nfp64, sizeof(h), cudaMemcpyDeviceToHost));
    if ((int)h[2]) return fail(RKR_ETIMEOUT, "latency scan wait timed out (%d)", (int)h[2]);
  }
  if (offs_host[nq] > capacity)
    return fail(RKR_ENOMEM, "candidate capacity %lld is below the %lld candidates found",
                (long long)capacity, (long long)offs_host[nq]);
  return RKR_OK;
}

rkr_status run_query_approx_single(const rkr_index *idx, const QueryCommon &qc, int nq, double c,
                                   int32_t *users_d, uint32_t *nlo_d, uint32_t *nup_d,
                                   double *est_d, int32_t *case_d, int32_t *nc_d,
                                   rkr_query_stats *stats, cudaStream_t st) {
  const int64_t n = idx->n;
  DevBuf bs[7], b7, b8, b9, b10, b11;
  ScanBufs sb;
  RKR_TRY(alloc_scan(idx, nq, tuning().latency_ctas_per_sm, bs, sb, st));
  uint32_t *clo, *cup;
  int32_t *cu, *cj;
  double *cth;
  RKR_TRY(tmp_alloc(b7, &cu, n, st));
  RKR_TRY(tmp_alloc(b8, &clo, n, st));
  RKR_TRY(tmp_alloc(b9, &cup, n, st));
  RKR_TRY(tmp_alloc(b10, &cj, n, st));
  RKR_TRY(tmp_alloc(b11, &cth, n, st));
  int *err = (int *)(sb.nfp64 + 1);
  const unsigned cgrid = (unsigned)((n + 1023) / 1024);   // four users a thread
  double ms = 0.0;
  SpanClock clk(st);
  const int t1 = clk.begin(&ms);
  for (int q = 0; q < nq; ++q) {
    RKR_TRY(scan_pass(idx, qc, q, sb, st));
    {
      const int prof_slot = prof_begin("k_latency_compact", st);
      k_latency_compact<<<cgrid, 256, 0, st>>>(n, sb.nlo, sb.nup, sb.jall, sb.T, q, sb.qcount, cu,
                                               clo, cup, cj, cth);
      prof_end(prof_slot, st, 0.0);
      note_launch();
    }
    RKR_TRY(launch_select_approx(q, 1, qc.out_off_d, sb.qcount, cu, clo, cup, cth, cj, qc.Qd,
                                 qc.kq_d, c, qc.out_off_d, users_d, nlo_d, nup_d, est_d, case_d,
                                 nc_d, err, st, idx));
  }
  RKR_CUDA(cudaGetLastError());
  clk.end(t1);
  unsigned long long h[3] = {0, 0, 0};
  RKR_CUDA(cudaMemcpyAsync(h, sb.nfp64, sizeof(h), cudaMemcpyDeviceToHost, st));
  RKR_CUDA(cudaStreamSynchronize(st));
  clk.finish();
  if ((int)h[2]) return fail(RKR_ETIMEOUT, "latency scan wait timed out (%d)", (int)h[2]);
  if ((int)h[1]) return fail(RKR_EINTERNAL, "fewer than k candidates for a query");
  if (stats) {
    stats->pairs = n * (int64_t)nq;
    stats->candidates = 0;
    stats->fp64_dots = (int64_t)h[0];
    stats->ms_theta = ms;
  }
  return RKR_OK;
}

}  // namespace rkr

// ------------------------------------------------------------------ session
// A serving form of the one-at-a-time path: persistent device buffers for one
// query and a CUDA graph of its launches (scan with the cut, compaction, steps 2-3),
// captured once at creation and replayed per query.
struct rkr_session {
  rkr_index *idx = nullptr;
  int max_k = 0, d = 0;
  double c = 2.0;
  cudaStream_t st = nullptr;
  unsigned char *in_dev = nullptr;   // an In
  int64_t *off_dev = nullptr;
  // outputs (pinned host memory, max_k entries each) and error words
  double *oest = nullptr;
  int32_t *users = nullptr, *ocase = nullptr, *onc = nullptr;
  int32_t *oerr = nullptr;   // [0] selection, [1] scan
  uint32_t *onlo = nullptr, *onup = nullptr;
  rkr::DevBuf scan_bufs[7], cand_bufs[5], out_bufs[2];
  rkr::lat::ScanBufs sb;
  uint32_t *clo = nullptr, *cup = nullptr;
  int32_t *cu = nullptr, *cj = nullptr;
  double *cth = nullptr;
  // pinned host memory: the query with its norm bound and k as one block, copied to
  // in_dev by the graph; the outputs and the two error words, written by the kernels
  struct In {
    float q[rkr::kMaxD];
    float qn;
    int32_t k;
    uint32_t wait;   // stage wait limit of the bulk-staged scan
  };
  In *in_h = nullptr;
  unsigned char *out_h = nullptr;
  cudaGraph_t graph = nullptr;
  cudaGraphExec_t exec = nullptr;
};

namespace rkr {
namespace {

rkr_status session_enqueue(rkr_session *s) {
  QueryCommon qc;
  qc.Qd = (float *)(s->in_dev + offsetof(rkr_session::In, q));
  qc.qnrm = (float *)(s->in_dev + offsetof(rkr_session::In, qn));
  qc.kq_d = (int32_t *)(s->in_dev + offsetof(rkr_session::In, k));
  qc.out_off_d = s->off_dev;
  qc.bf = s->idx->binfp;
  qc.xbf = s->idx->xbin;
  RKR_CUDA(cudaMemcpyAsync(s->in_dev, s->in_h, sizeof(rkr_session::In), cudaMemcpyHostToDevice,
                           s->st));
  RKR_TRY(scan_pass(s->idx, qc, 0, s->sb, s->st));
  const int64_t n = s->idx->n;
  const unsigned cgrid = (unsigned)((n + 1023) / 1024);   // four users a thread
  k_latency_compact<<<cgrid, 256, 0, s->st>>>(n, s->sb.nlo, s->sb.nup, s->sb.jall, s->sb.T, 0,
                                              s->sb.qcount, s->cu, s->clo, s->cup, s->cj,
                                              s->cth);
  note_launch();
  RKR_TRY(launch_select_approx(0, 1, s->off_dev, s->sb.qcount, s->cu, s->clo, s->cup, s->cth,
                               s->cj, qc.Qd, qc.kq_d, s->c, s->off_dev, s->users, s->onlo,
                               s->onup, s->oest, s->ocase, s->onc, s->oerr, s->st, s->idx));
  return RKR_OK;
}

void session_release(rkr_session *s) {
  if (!s) return;
  if (s->exec) cudaGraphExecDestroy(s->exec);
  if (s->graph) cudaGraphDestroy(s->graph);
  // device blocks go back to the pool on the session's stream, before it goes
  for (DevBuf *group : {s->scan_bufs, s->cand_bufs, s->out_bufs}) {
    const int count = group == s->scan_bufs ? 7 : (group == s->cand_bufs ? 5 : 2);
    for (int i = 0; i < count; ++i)
      if (group[i].p) {
        cudaFreeAsync(group[i].p, group[i].st);
        group[i].p = nullptr;
      }
  }
  if (s->st) {
    cudaStreamSynchronize(s->st);
    cudaStreamDestroy(s->st);
  }
  if (s->in_h) cudaFreeHost(s->in_h);
  if (s->out_h) cudaFreeHost(s->out_h);
  delete s;
}

}  // namespace
}  // namespace rkr

using namespace rkr;

extern "C" rkr_status rkr_session_create(rkr_index *idx, int32_t max_k, double c, void *stream,
                                         rkr_session **out) {
  set_error("%s", "");
  if (!idx || !out) return fail(RKR_EINVAL, "null argument");
  *out = nullptr;
  if (max_k < 1 || max_k > kMaxK || max_k > idx->n)
    return fail(RKR_EINVAL, "max_k must be in [1, min(n, %d)]", kMaxK);
  if (!(c >= 1.0) || !isfinite(c)) return fail(RKR_EINVAL, "c must be a finite value >= 1");
  RKR_TRY(check_device());
  rkr_session *s = new (std::nothrow) rkr_session();
  if (!s) return fail(RKR_ENOMEM, "host allocation failed");
  struct Guard {
    rkr_session *s;
    ~Guard() { session_release(s); }
  } guard{s};
  s->idx = idx;
  s->max_k = max_k;
  s->c = c;
  s->d = idx->d;
  RKR_CUDA(cudaStreamCreateWithFlags(&s->st, cudaStreamNonBlocking));
  (void)stream;  // the session keeps its own stream: the graph is captured on it
  cudaStream_t st = s->st;
  const int64_t n = idx->n;
  RKR_TRY(alloc_scan(idx, 1, tuning().latency_ctas_per_sm, s->scan_bufs, s->sb, st));
  RKR_TRY(tmp_alloc(s->cand_bufs[0], &s->cu, n, st));
  RKR_TRY(tmp_alloc(s->cand_bufs[1], &s->clo, n, st));
  RKR_TRY(tmp_alloc(s->cand_bufs[2], &s->cup, n, st));
  RKR_TRY(tmp_alloc(s->cand_bufs[3], &s->cj, n, st));
  RKR_TRY(tmp_alloc(s->cand_bufs[4], &s->cth, n, st));
  RKR_TRY(tmp_alloc(s->out_bufs[0], &s->in_dev, sizeof(rkr_session::In), st));
  RKR_TRY(tmp_alloc(s->out_bufs[1], &s->off_dev, 2, st));
  RKR_CUDA(cudaMemsetAsync(s->off_dev, 0, 2 * sizeof(int64_t), st));
  const size_t K = (size_t)max_k;
  const size_t out_bytes = K * (8 + 4 + 4 + 4) + 4 * sizeof(int32_t);
  RKR_CUDA(cudaMallocHost(&s->in_h, sizeof(rkr_session::In)));
  memset(s->in_h, 0, sizeof(rkr_session::In));
  s->in_h->k = 1;
  s->in_h->wait = epi_wait_limit();
  RKR_CUDA(cudaMallocHost(&s->out_h, out_bytes));
  memset(s->out_h, 0, out_bytes);
  s->oest = (double *)s->out_h;
  s->users = (int32_t *)(s->out_h + 8 * K);
  s->onlo = (uint32_t *)(s->out_h + 12 * K);
  s->onup = (uint32_t *)(s->out_h + 16 * K);
  s->ocase = (int32_t *)(s->out_h + 20 * K);
  s->onc = s->ocase + 1;
  s->oerr = s->ocase + 2;
  s->sb.err = s->oerr + 1;
  s->sb.wait_p = (const uint32_t *)(s->in_dev + offsetof(rkr_session::In, wait));
  // one uncaptured run (sets function attributes, warms the pool), then the capture
  RKR_TRY(session_enqueue(s));
  RKR_CUDA(cudaStreamSynchronize(st));
  RKR_CUDA(cudaStreamBeginCapture(st, cudaStreamCaptureModeThreadLocal));
  const rkr_status es = session_enqueue(s);
  cudaGraph_t g = nullptr;
  const cudaError_t ce = cudaStreamEndCapture(st, &g);
  s->graph = g;
  RKR_TRY(es);
  if (ce != cudaSuccess) return cuda_fail(ce, "cudaStreamEndCapture");
  RKR_CUDA(cudaGraphInstantiate(&s->exec, s->graph, 0));
  *out = s;
  guard.s = nullptr;
  return RKR_OK;
}

extern "C" rkr_status rkr_session_query(rkr_session *s, const float *q, int32_t k,
                                        int32_t *out_users, uint32_t *out_nlow,
                                        uint32_t *out_nup, double *out_est, int32_t *out_case,
                                        int32_t *out_nc) {
  set_error("%s", "");
  if (!s || !q || !out_users) return fail(RKR_EINVAL, "null argument");
  if (k < 1 || k > s->max_k) return fail(RKR_EINVAL, "k must be in [1, %d]", s->max_k);
  const int d = s->d;
  cudaStream_t st = s->st;
  cudaPointerAttributes pa;
  const bool qdev = cudaPointerGetAttributes(&pa, q) == cudaSuccess &&
                    (pa.type == cudaMemoryTypeDevice || pa.type == cudaMemoryTypeManaged);
  cudaGetLastError();
  float *qh = s->in_h->q;
  if (qdev) RKR_CUDA(cudaMemcpy(qh, q, sizeof(float) * d, cudaMemcpyDeviceToHost));
  else memcpy(qh, q, sizeof(float) * d);
  double ss = 0.0;
  for (int i = 0; i < d; ++i) {
    if (!isfinite(qh[i])) return fail(RKR_EINVAL, "q must be finite");
    ss += (double)qh[i] * (double)qh[i];
  }
  if (sqrt(ss) * (1.0 + 0x1p-20) > (double)s->idx->pmax) {
    // outside the item norms: the general call, whose bounds need no assumption about
    // the query's norm (the scan itself makes none: see TightBins)
    return rkr_query_approx_single(s->idx, q, 1, &k, s->c, out_users, out_nlow, out_nup,
                                   out_est, out_case, out_nc, nullptr, st);
  }
  // FP32 upper bound of ||q||, as row_norms forms it on the device
  const double nv = sqrt(ss) * (1.0 + 0x1p-40) + 1e-300;
  float qn = (float)nv;
  if ((double)qn < nv) qn = nextafterf(qn, INFINITY);
  s->in_h->qn = qn;
  s->in_h->k = k;
  s->in_h->wait = epi_wait_limit();
  s->oerr[0] = s->oerr[1] = 0;
  RKR_CUDA(cudaGraphLaunch(s->exec, st));
  RKR_CUDA(cudaStreamSynchronize(st));
  if (s->oerr[1]) return fail(RKR_ETIMEOUT, "latency scan wait timed out (%d)", s->oerr[1]);
  if (s->oerr[0]) return fail(RKR_EINTERNAL, "fewer than k candidates for the query");
  const size_t K = (size_t)k;
  struct Out {
    void *dst;
    const void *src;
    size_t bytes;
  } outs[] = {{out_users, s->users, 4 * K}, {out_nlow, s->onlo, 4 * K}, {out_nup, s->onup, 4 * K},
              {out_est, s->oest, 8 * K},    {out_case, s->ocase, 4},    {out_nc, s->onc, 4}};
  for (const Out &x : outs) {
    if (!x.dst) continue;
    cudaPointerAttributes a;
    const bool dev = cudaPointerGetAttributes(&a, x.dst) == cudaSuccess &&
                     (a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged);
    cudaGetLastError();
    if (dev) RKR_CUDA(cudaMemcpy(x.dst, x.src, x.bytes, cudaMemcpyHostToDevice));
    else memcpy(x.dst, x.src, x.bytes);
  }
  return RKR_OK;
}

extern "C" void rkr_session_free(rkr_session *s) { session_release(s); }
