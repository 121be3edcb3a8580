// query.cu -- query processing for both paths.
//
// Both paths share one plan.  For every user u the index holds a table of
// rank bounds on the threshold grid t_1..t_tau of u (the sampled table N of
// Alg. 1 for the c-approximate path; the exact count bounds XLO/XHI for the
// exact path) and two level tables JU/JL that turn a bin j into the rank level
// 2^L the table implies.  A query batch is processed as
//   pass 1  u.q screened for every (u, q) -> bin interval [jlo, jhi] ->
//           per-query histograms of the upper-bound level and the lower-bound level
//   cutoff  L*(q) = smallest level holding k upper bounds: R_up_k (approximate
//           path) or the k-th smallest rank (exact path) is at most 2^L* on the scale
//   pass 2  u.q screened again; users whose lower bound may reach 2^L* are
//           written to the candidate list of q (all others provably cannot matter)
//   resolve canonical FP64 u.q for each candidate; exact bin and table values
//           (approximate) or an exact recount of the rank over P (exact)
//   select  one CTA per query: Section 4.3 steps 1-3 (approximate) or the k
//           smallest (rank, index) (exact) over the candidates.
#include <math.h>
#include <stdlib.h>
#include <string.h>

#include <algorithm>

#include <vector>

#include "index.cuh"
#include "sort.cuh"
#include "select.cuh"
#include "simt.cuh"
#include "tcops.cuh"

namespace rkr {


// Cutoff level of each query: L* = the smallest level holding k upper bounds;
// below = pairs whose upper bound lies in a lower level; ncand = pairs whose
// lower bound lies in a level <= L* (an upper bound of the candidate count).
// Only levels <= lcap are complete in the histograms; a query that does not
// reach k there gets L* = kDeep and is screened again without skipping.
constexpr int kDeep = kMaxLevels;

__global__ void k_cutoff(int nq, const uint32_t *__restrict__ hist_up,
                         const uint32_t *__restrict__ hist_lo, const int32_t *__restrict__ kq,
                         int nlev, int lcap, int32_t *__restrict__ lstar,
                         uint64_t *__restrict__ below, int64_t *__restrict__ ncand) {
  int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= nq) return;
  uint64_t cum = 0, prev = 0;
  int L = lcap >= nlev - 1 ? nlev - 1 : kDeep;
  const int lend = lcap < 31 ? lcap : 31;
  for (int l = 0; l <= lend; ++l) {
    prev = cum;
    cum += hist_up[(int64_t)q * 32 + l];
    if (cum >= (uint64_t)kq[q]) { L = l; break; }
  }
  if (L == kDeep) {
    lstar[q] = kDeep;
    below[q] = 0;
    ncand[q] = 0;
    return;
  }
  if (L > nlev - 1) L = nlev - 1;
  uint64_t c = 0;
  for (int l = 0; l <= L; ++l) c += hist_lo[(int64_t)q * 32 + l];
  lstar[q] = L;
  below[q] = prev;
  ncand[q] = (int64_t)c;
}

// Skip score of each user for skip level LS: the largest float x such that every
// screened upper end x_hi <= x gives a bin upper bound j_hi < JL[LS], so the
// pair's lower bound lies above level LS.  -inf when no such x is found.
__global__ void k_skip_scores(int64_t n, const BinFP *__restrict__ bf,
                              const int16_t *__restrict__ JL, int LS, float *__restrict__ xs) {
  int64_t u = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (u >= n) return;
  const int J = JL[u * kMaxLevels + LS];
  const BinFP b = bf[u];
  float x = -INFINITY;
  if (J >= 1 && b.invd32 > 0.0f && !(b.err > 1e6f)) {
    // bin_vhi(x) < J - 1 gives floor(v) + 1 <= J - 1
    const float target = (float)(J - 1);
    double x0 = (double)b.fmin32 + ((double)target - (double)b.err - 1.0) / (double)b.invd32;
    float c = __double2float_rd(x0);
    for (int it = 0; it < 64 && !(bin_vhi(b, c) < target); ++it) c = nextafterf(c, -INFINITY);
    if (bin_vhi(b, c) < target) x = c;
  }
  xs[u] = x;
}

// Rows of the deep queries, gathered for their own screening launches.
__global__ void k_gather_qrows(int nd, const int32_t *__restrict__ rows, int kp, int ld,
                               const __nv_bfloat16 *__restrict__ hi,
                               const __nv_bfloat16 *__restrict__ lo,
                               const tc::RowBound *__restrict__ rb1,
                               const tc::RowBound *__restrict__ rb3,
                               __nv_bfloat16 *__restrict__ ohi, __nv_bfloat16 *__restrict__ olo,
                               tc::RowBound *__restrict__ orb1, tc::RowBound *__restrict__ orb3,
                               uint32_t *__restrict__ hist, int nq) {
  const int i = blockIdx.x;
  if (i >= nd) return;
  const int64_t r = rows[i];
  for (int k = threadIdx.x; k < kp; k += blockDim.x) {
    ohi[(int64_t)i * ld + k] = hi[r * ld + k];
    olo[(int64_t)i * ld + k] = lo[r * ld + k];
  }
  if (threadIdx.x < 32) {  // the histograms of the skipping pass are incomplete
    hist[r * 32 + threadIdx.x] = 0;
    hist[((int64_t)nq + r) * 32 + threadIdx.x] = 0;
  }
  if (threadIdx.x == 0) {
    orb1[i] = rb1[r];
    orb3[i] = rb3[r];
  }
}

// Refined cap: the upper edge of the fine bucket of level L* where the running
// count of upper bounds reaches k; the k-th smallest upper bound is <= cap.
__global__ void k_cutoff_fine(int nq, const uint32_t *__restrict__ fine,
                              const uint64_t *__restrict__ below, const int32_t *__restrict__ lstar,
                              const int32_t *__restrict__ kq, uint32_t scale,
                              uint32_t *__restrict__ cap) {
  int q = blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= nq) return;
  const int L = lstar[q];
  uint64_t hi = level_bound(L, scale);
  uint64_t base = L == 0 ? 0 : level_bound(L - 1, scale) + 1;
  uint64_t width = (hi - base + 1024) / 1024;
  uint64_t cum = below[q], c = hi;
  for (int b = 0; b < 1024; ++b) {
    cum += fine[(int64_t)q * 1024 + b];
    if (cum >= (uint64_t)kq[q]) { c = base + (uint64_t)(b + 1) * width - 1; break; }
  }
  if (c > hi) c = hi;
  cap[q] = (uint32_t)(c > 0xffffffffull ? 0xffffffffull : c);
}

// --------------------------------------------------------- approximate path

__global__ void k_resolve_approx(int64_t count, const int32_t *__restrict__ cu,
                                 const int32_t *__restrict__ cq, const float *__restrict__ cx,
                                 const tc::RowBound *__restrict__ urb,
                                 const tc::RowBound *__restrict__ qrb, tc::Gacc gacc, float gcan,
                                 const float *__restrict__ U, const float *__restrict__ Q, int d,
                                 const double *__restrict__ fmin,
                                 const double *__restrict__ delta, const BinFP *__restrict__ bf,
                                 const uint32_t *__restrict__ N,
                                 int tau, uint32_t top, double *__restrict__ th,
                                 int32_t *__restrict__ cj, uint32_t *__restrict__ nlo,
                                 uint32_t *__restrict__ nup,
                                 unsigned long long *__restrict__ nfp64) {
  int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= count) return;
  int64_t u = cu[i];
  if (u < 0) return;  // unused slot at the end of a query's segment
  int q = cq[i];
  const float *uu = U + u * d, *qq = Q + (int64_t)q * d;
  // j from the screened score and its bound when both ends fall in one bin (no
  // row is read); else from the compensated interval of u.q; else from the
  // canonical u.q.  u.q itself is formed later, only for the users whose step-3
  // estimate is needed (NaN marks it as not yet formed).
  int jlo = 0, jhi = tau;
  const float x = cx[i];
  if (x == x) {   // NaN: the candidate has no screened score
    const float b = tc::screen_bound_tc(urb[u], qrb[q], gacc, gcan);
    bin_interval(bf[u], fmin[u], tau, __fsub_rd(x, b), __fadd_ru(x, b), jlo, jhi);
  }
  if (jlo != jhi) {
    float tlo, thi;
    dot2_interval_f(uu, qq, d, tlo, thi);
    bin_interval(bf[u], fmin[u], tau, tlo, thi, jlo, jhi);
  }
  int j;
  if (jlo == jhi) {
    j = jlo;
    th[i] = __longlong_as_double(0x7ff8000000000000ll);
  } else {
    const double theta = canon_dot(uu, qq, d);
    j = exact_j(theta, fmin[u], delta[u], tau);
    th[i] = theta;
    atomicAdd(nfp64, 1ull);
  }
  cj[i] = j;
  nlo[i] = j < tau ? N[u * tau + j] : 0u;
  nup[i] = j >= 1 ? N[u * tau + j - 1] : top;
}

struct ApproxCand {
  const int32_t *uid;
  const uint32_t *nlo, *nup;
  double *th;          // canonical u.q (NaN: not formed); overwritten by estimates
  const int32_t *j;
  const float *U, *Q;  // rows, for forming u.q on demand
  int d;
  unsigned long long *nfp64;   // canonical products formed (may be null)
};

// Width of a radix key for counts up to `top`: a multiple of 8 bits whose largest
// value lies above top (it stands for the dropped candidates' ~0, see count_key).
__host__ __device__ inline int count_bits(uint64_t top) {
  int bits = 8;
  while (bits < 32 && (((uint64_t)1 << bits) - 1) <= top) bits += 8;
  return bits;
}
__device__ __forceinline__ uint64_t count_key(uint32_t c, int bits) {
  return bits < 32 ? min(c, (1u << bits) - 1u) : c;
}

// Bytes of a user index, in bits.
static int user_bits(int64_t n) {
  int bits = 8;
  while (bits < 32 && ((int64_t)1 << bits) < n) bits += 8;
  return bits;
}

// Threads of the per-query selections: 256 where many queries share the SMs, 1,024
// where there are fewer queries than SMs (one CTA's walk of its candidates is then
// the time of the launch).
constexpr int kSelThreads = 256;
constexpr int kSelThreadsFew = 1024;
constexpr int kSelSmall = 512;     // entries sorted beside the survivors (k_select_approx)
constexpr size_t kSelSmem = sizeof(SortEnt) * (kMaxK + kSelSmall);
// Rows staged at a time for the canonical products of k_select_approx with 1,024
// threads, behind the query as doubles.
constexpr int kSelRows = 128;
static size_t select_smem(bool few, int d) {
  return kSelSmem + (few ? sizeof(double) * d + sizeof(float) * kSelRows * (d | 1) : 0);
}

// Entries a selection may leave to the sort: 64, which its short form places at once,
// or as many as the bitonic form sorts for k.
__device__ __forceinline__ uint32_t sort_room(int k) {
  uint32_t r = 64;
  while (r < (uint32_t)k) r <<= 1;
  return r;
}

// One CTA per query: steps 1-3 of Section 4.3 over the query's candidates.
template <int THREADS>
__global__ void __launch_bounds__(THREADS)
    k_select_approx(int qa, const int64_t *__restrict__ qoff, const uint32_t *__restrict__ qcount,
                    ApproxCand C,
                    const int32_t *__restrict__ kq, double c, uint32_t s, int tau,
                    const double *__restrict__ fmin, const double *__restrict__ delta,
                    const int64_t *__restrict__ out_off, int32_t *__restrict__ out_users,
                    uint32_t *__restrict__ out_nlo, uint32_t *__restrict__ out_nup,
                    double *__restrict__ out_est, int32_t *__restrict__ out_case,
                    int32_t *__restrict__ out_nc, int *__restrict__ err, uint32_t top,
                    int ubits) {
  extern __shared__ unsigned char sbuf[];
  SortEnt *ent = (SortEnt *)sbuf;                   // kMaxK entries
  SortEnt *small = ent + kMaxK;                     // kSelSmall entries
  __shared__ __align__(16) uint32_t hist[512];
  __shared__ uint64_t bc[4];
  __shared__ unsigned long long cnt_acc;
  __shared__ int gcount;
  const int q = qa + blockIdx.x;
  const int64_t base = qoff[q] - qoff[qa];
  const int64_t cnt = qcount[q];
  const int k = kq[q];
  if (cnt < k) {  // cannot happen when the screening passes are consistent
    if (threadIdx.x == 0) atomicExch(err, 1);
    return;
  }
  const int32_t *uid = C.uid + base;
  const uint32_t *nlo = C.nlo + base, *nup = C.nup + base;
  double *th = C.th + base;
  const int32_t *cj = C.j + base;
  const float *qrow = C.Q + (int64_t)q * C.d;
  // Step-3 estimate from the canonical u.q: some 40 FP64 operations and, where u.q
  // is not formed yet, a canonical product, so each candidate's is formed once.
  auto est_of = [&](int64_t i) {
    int32_t u = uid[i];
    double t = th[i];
    if (t != t) {  // not formed yet
      t = canon_dot(C.U + (int64_t)u * C.d, qrow, C.d);
      if (C.nfp64) atomicAdd(C.nfp64, 1ull);
    }
    return interp_est(t, cj[i], nlo[i], nup[i], fmin[u], delta[u], tau, s);
  };
  // Canonical products of the users of e[0, count) that have none yet, where few
  // queries leave the SM to this one: their rows are staged in shared memory by the
  // whole block (one round trip to memory for 128 of them), then a lane per row adds
  // its products in order, with operands converted by integer operations.  A lane
  // reading its own row from memory took 245 cycles a dimension for 32 users, this 115 to 145
  // (an FP64 instruction alone takes 76).
  auto form_dots = [&](const SortEnt *e, int count) {
    if constexpr (THREADS == kSelThreadsFew) {
      double *qd = (double *)(small + kSelSmall);
      float *tile = (float *)(qd + C.d);
      const int d = C.d, ld = d | 1, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
      for (int c0 = threadIdx.x; c0 < d; c0 += THREADS) qd[c0] = exact_double(qrow[c0]);
      for (int b = 0; b < count; b += kSelRows) {
        const int nr = min(kSelRows, count - b);
        __syncthreads();
        for (int r = warp; r < nr; r += THREADS / 32) {
          const int64_t i = e[b + r].idx;
          const double t = th[i];
          if (t == t) continue;
          const float *row = C.U + (int64_t)uid[i] * d;
          float v[kMaxD / 32];
#pragma unroll
          for (int p = 0; p < kMaxD / 32; ++p) v[p] = lane + 32 * p < d ? row[lane + 32 * p] : 0.0f;
#pragma unroll
          for (int p = 0; p < kMaxD / 32; ++p)
            if (lane + 32 * p < d) tile[r * ld + lane + 32 * p] = v[p];
        }
        __syncthreads();
        if (threadIdx.x < nr) {
          const int64_t i = e[b + threadIdx.x].idx;
          const double t = th[i];
          if (t != t) {
            const float *x = tile + threadIdx.x * ld;
            double acc = 0.0;
#pragma unroll 8
            for (int c0 = 0; c0 < d; ++c0) acc = __fma_rn(exact_double(x[c0]), qd[c0], acc);
            th[i] = acc;
            if (C.nfp64) atomicAdd(C.nfp64, 1ull);
          }
        }
      }
      __syncthreads();
    }
  };
  // Step 1: k-th smallest lower and upper bound numerators (at most top).
  const int nbits = count_bits(top);
  uint64_t Rlo, Rup;
  block_kth_pair(nlo, nup, cnt, (uint64_t)k, nbits, hist, bc, Rlo, Rup);
  // c R_low_k against R_up_k, by one thread: an FP64 instruction of every warp of the
  // block takes eight times as long
  if (threadIdx.x == 0) {
    const double lhs = c * (double)((uint64_t)s + Rlo);
    bc[0] = lhs >= (double)((uint64_t)s + Rup);
    bc[1] = (uint64_t)floor(lhs);
  }
  __syncthreads();
  const bool caseA = bc[0] != 0;
  const uint64_t lim = bc[1];
  __syncthreads();   // bc is the selections' from here on
  const int64_t obase = out_off[q];
  int nc;
  if (caseA) {
    // k smallest (r_up, r_low, index).  All with nup <= Rup are gathered; if they are
    // few, sorting them gives the k first.  Otherwise all with nup < Rup, then of the
    // ties the smallest (nlo, index).
    auto put = [&](int pos, int64_t i) {
      ent[pos].k1 = ((uint64_t)nup[i] << 32) | nlo[i];
      ent[pos].k2 = (uint32_t)uid[i];
      ent[pos].idx = (int32_t)i;
    };
    const uint32_t room = sort_room(k);
    if (threadIdx.x == 0) {
      gcount = 0;
      cnt_acc = 0;
    }
    __syncthreads();
    for (int64_t i0 = 0; i0 < cnt; i0 += blockDim.x) {   // whole warps
      const int64_t i = i0 + threadIdx.x;
      const uint64_t v = i < cnt ? nup[i] : ~0ull;
      if (v <= Rup) {
        const int pos = atomicAdd(&gcount, 1);
        if (pos < (int)room) put(pos, i);
      }
      const unsigned less = __ballot_sync(0xffffffffu, v < Rup);
      if ((threadIdx.x & 31) == 0 && less) atomicAdd(&cnt_acc, (unsigned long long)__popc(less));
    }
    __syncthreads();
    const int upto = gcount;
    const int64_t below = (int64_t)cnt_acc;
    __syncthreads();
    if (upto > (int)room) {
      // (below < k: Rup is the k-th; the keys are distinct, so at most `room` remain)
      auto tie_key = [&](int64_t i) { return ((uint64_t)nlo[i] << ubits) | (uint32_t)uid[i]; };
      uint32_t ties;
      const uint64_t last = block_kth_cut(cnt, (uint64_t)(k - below), nbits + ubits,
                                          [&](int64_t i, uint64_t &key) {
                                            key = tie_key(i);
                                            return (uint64_t)nup[i] == Rup;
                                          },
                                          hist, bc, room - (uint32_t)below, ties);
      if (threadIdx.x == 0) gcount = 0;
      __syncthreads();
      for (int64_t i = threadIdx.x; i < cnt; i += blockDim.x) {
        const uint64_t a = nup[i];
        if (a < Rup || (a == Rup && tie_key(i) <= last)) {
          const int pos = atomicAdd(&gcount, 1);
          if (pos < kMaxK) put(pos, i);
        }
      }
    }
    __syncthreads();
    int got = min(gcount, kMaxK);
    block_sort(ent, got);
    if (out_est) form_dots(ent, min(got, k));
    for (int r = threadIdx.x; r < got && r < k; r += blockDim.x) {
      int64_t i = ent[r].idx;
      out_users[obase + r] = uid[i];
      if (out_nlo) out_nlo[obase + r] = nlo[i];
      if (out_nup) out_nup[obase + r] = nup[i];
      if (out_est) out_est[obase + r] = est_of(i);
    }
    nc = k;
  } else {
    // U_c = {r_up <= c R_low_k}: fewer than k users, (r_up, r_low, index) order
    // s + nup <= c (s + R_low_k): integers (below 2^53) against a real, so against
    // its floor
    auto in_c = [&](int64_t i) { return (uint64_t)s + nup[i] <= lim; };
    if (threadIdx.x == 0) gcount = 0;
    __syncthreads();
    for (int64_t i = threadIdx.x; i < cnt; i += blockDim.x) {
      if (in_c(i)) {
        int pos = atomicAdd(&gcount, 1);
        if (pos < kMaxK) {
          ent[pos].k1 = ((uint64_t)nup[i] << 32) | nlo[i];
          ent[pos].k2 = (uint32_t)uid[i];
          ent[pos].idx = (int32_t)i;
        }
      }
    }
    __syncthreads();
    nc = min(gcount, kMaxK);
    block_sort(ent, nc);
    if (out_est) form_dots(ent, nc);
    for (int r = threadIdx.x; r < nc; r += blockDim.x) {
      int64_t i = ent[r].idx;
      out_users[obase + r] = uid[i];
      if (out_nlo) out_nlo[obase + r] = nlo[i];
      if (out_nup) out_nup[obase + r] = nup[i];
      if (out_est) out_est[obase + r] = est_of(i);
    }
    __syncthreads();
    // Step 3: survivors r_low <= R_up_k outside U_c, smallest (r_hat, index).  They
    // are gathered in shared memory first, so that their estimates are formed in
    // full warps; where they fit, the selection runs there, else over all candidates
    // with the estimates in the place of u.q in th.
    auto in_t = [&](int64_t i) { return (uint64_t)nlo[i] <= Rup && !in_c(i); };
    const int need = k - nc;
    if (threadIdx.x == 0) gcount = 0;
    __syncthreads();
    for (int64_t i = threadIdx.x; i < cnt; i += blockDim.x) {
      if (!in_t(i)) continue;
      const int pos = atomicAdd(&gcount, 1);
      if (pos < kMaxK) ent[pos].idx = (int32_t)i;
      else th[i] = est_of(i);
    }
    __syncthreads();
    const int nt = gcount;
    __syncthreads();   // every thread has the count before it is reset
    const bool fits = nt <= kMaxK && need <= kSelSmall;
    form_dots(ent, min(nt, kMaxK));
    for (int e = threadIdx.x; e < min(nt, kMaxK); e += blockDim.x) {
      const int64_t i = ent[e].idx;
      const double est = est_of(i);
      ent[e].k1 = dkey(est);
      ent[e].k2 = (uint32_t)uid[i];
      if (!fits) th[i] = est;
    }
    if (threadIdx.x == 0) gcount = 0;
    __syncthreads();
    if (fits) {
      // those up to the need-th estimate, or a little past it, go to the sort; only
      // estimates that tie beyond its room are told apart by their users
      const uint32_t room = sort_room(need);
      uint64_t ke = ~0ull, ku = ~0ull;
      uint32_t upto = (uint32_t)nt;
      if (upto > room)
        ke = block_kth_cut(nt, (uint64_t)need, 64,
                           [&](int64_t e, uint64_t &key) {
                             key = ent[e].k1;
                             return true;
                           },
                           hist, bc, room, upto);
      if (upto > room) {
        const int64_t below =
            block_count(nt, [&](int64_t e) { return ent[e].k1 < ke; }, &cnt_acc);
        ku = block_kth(nt, (uint64_t)(need - below), 32,
                       [&](int64_t e, uint64_t &key) {
                         key = ent[e].k2;
                         return ent[e].k1 == ke;
                       },
                       hist, bc);
      }
      for (int e = threadIdx.x; e < nt; e += blockDim.x) {
        const SortEnt x = ent[e];
        if (x.k1 < ke || (x.k1 == ke && (uint64_t)x.k2 <= ku)) {
          const int pos = atomicAdd(&gcount, 1);
          if (pos < kSelSmall) small[pos] = x;
        }
      }
      __syncthreads();
      const int got = min(gcount, kSelSmall);
      block_sort(small, got);
      for (int r = threadIdx.x; r < got && r < need; r += blockDim.x) {
        const int64_t i = small[r].idx;
        out_users[obase + nc + r] = uid[i];
        if (out_nlo) out_nlo[obase + nc + r] = nlo[i];
        if (out_nup) out_nup[obase + nc + r] = nup[i];
        if (out_est) out_est[obase + nc + r] = __longlong_as_double((long long)small[r].k1);
      }
    } else {
    uint64_t ke = block_kth(cnt, (uint64_t)need, 64,
                            [&](int64_t i, uint64_t &key) {
                              if (!in_t(i)) return false;
                              key = dkey(th[i]);
                              return true;
                            },
                            hist, bc);
    int64_t below = block_count(cnt, [&](int64_t i) { return in_t(i) && dkey(th[i]) < ke; },
                                &cnt_acc);
    uint64_t ku = ~0ull;
    if (below < need)
      ku = block_kth(cnt, (uint64_t)(need - below), 32,
                     [&](int64_t i, uint64_t &key) {
                       if (!in_t(i) || dkey(th[i]) != ke) return false;
                       key = (uint32_t)uid[i];
                       return true;
                     },
                     hist, bc);
    if (threadIdx.x == 0) gcount = 0;
    __syncthreads();
    for (int64_t i = threadIdx.x; i < cnt; i += blockDim.x) {
      if (!in_t(i)) continue;
      uint64_t ek = dkey(th[i]);
      if (ek < ke || (ek == ke && (uint64_t)(uint32_t)uid[i] <= ku)) {
        int pos = atomicAdd(&gcount, 1);
        if (pos < kMaxK) {
          ent[pos].k1 = ek;
          ent[pos].k2 = (uint32_t)uid[i];
          ent[pos].idx = (int32_t)i;
        }
      }
    }
    __syncthreads();
    int got = min(gcount, kMaxK);
    block_sort(ent, got);
    for (int r = threadIdx.x; r < got && nc + r < k; r += blockDim.x) {
      int64_t i = ent[r].idx;
      out_users[obase + nc + r] = uid[i];
      if (out_nlo) out_nlo[obase + nc + r] = nlo[i];
      if (out_nup) out_nup[obase + nc + r] = nup[i];
      if (out_est) out_est[obase + nc + r] = __longlong_as_double((long long)ent[r].k1);
    }
    }
  }
  if (threadIdx.x == 0) {
    if (out_case) out_case[q] = caseA ? 1 : 2;
    if (out_nc) out_nc[q] = nc;
  }
}

// -------------------------------------------------------------- exact path

// Canonical u.q of each candidate and its sort key (user, order-preserving u.q).
__global__ void k_cand_theta(int64_t count, const int32_t *__restrict__ cu,
                             const int32_t *__restrict__ cq, const float *__restrict__ U,
                             const float *__restrict__ Q, int d, double *__restrict__ th,
                             uint64_t *__restrict__ key_hi, uint64_t *__restrict__ key_lo,
                             int32_t *__restrict__ val, int64_t Np2) {
  int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= Np2) return;
  if (i >= count || cu[i] < 0) {  // padding or an unused slot: sorted to the end
    key_hi[i] = ~0ull;
    key_lo[i] = ~0ull;
    val[i] = 0x7fffffff;
    return;
  }
  int64_t u = cu[i];
  double theta = canon_dot(U + u * d, Q + (int64_t)cq[i] * d, d);
  th[i] = theta;
  uint64_t bits = (uint64_t)__double_as_longlong(theta);
  key_hi[i] = (uint64_t)u;
  key_lo[i] = (bits >> 63) ? ~bits : (bits | 0x8000000000000000ull);
  val[i] = (int32_t)i;
}

// Segments of equal user in the sorted order: start index and length.  A user
// with fewer than seg_min thresholds (or every user, seg_min = 0) gets one
// segment per threshold; a longer run is cut into near-equal segments of at
// most kRecountSeg.  Segments
// of one threshold take slots from the front of [0, count), longer ones from
// the back, so that each kind is one range for its recount screen; seg_len of
// the slots between stays 0.
// nseg[0] = front slots, nseg[1] = distinct users, nseg[2] = back slots.
__global__ void k_segments(int64_t count, const uint64_t *__restrict__ key_hi, int seg_min,
                           unsigned long long *__restrict__ nseg, int64_t *__restrict__ seg_start,
                           int32_t *__restrict__ seg_len) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const bool first = i < count && key_hi[i] != ~0ull && (i == 0 || key_hi[i] != key_hi[i - 1]);
  int64_t e = i + 1;
  if (first)
    while (e < count && key_hi[e] == key_hi[i]) ++e;
  const int64_t run = first ? e - i : 0;
  const bool single = first && (seg_min == 0 || run < seg_min);
  // one atomic per warp for the distinct users and for the one-threshold slots
  // (a million candidates of one query would otherwise queue on one address)
  const int lane = threadIdx.x & 31;
  const unsigned nfirst = __popc(__ballot_sync(0xffffffffu, first));
  unsigned long long mine = single ? (unsigned long long)run : 0ull, incl = mine;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned long long t = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += t;
  }
  const unsigned long long tot = __shfl_sync(0xffffffffu, incl, 31);
  unsigned long long base = 0;
  if (lane == 31) {
    if (tot) base = atomicAdd(&nseg[0], tot);
    if (nfirst) atomicAdd(&nseg[1], (unsigned long long)nfirst);   // distinct users
  }
  base = __shfl_sync(0xffffffffu, base, 31);
  if (single) {   // one row per threshold
    const int64_t slot0 = (int64_t)(base + incl - mine);
    for (int64_t a = i; a < e; ++a) {
      seg_start[slot0 + (a - i)] = a;
      seg_len[slot0 + (a - i)] = 1;
    }
    return;
  }
  if (!first) return;
  // pieces of nearly equal length, at most kRecountSeg each
  const int64_t np = (run + kRecountSeg - 1) / kRecountSeg;
  for (int64_t p = 0; p < np; ++p) {
    const int64_t a = i + run * p / np, b = i + run * (p + 1) / np;
    const int64_t slot = count - 1 - (int64_t)atomicAdd(&nseg[2], 1ull);
    seg_start[slot] = a;
    seg_len[slot] = (int32_t)(b - a);
  }
}

// Per segment: its user, its thresholds in sorted order, and a zeroed histogram
// of L + 1 slots at hist[2 st0] (segments are disjoint since L >= 1).  A
// one-threshold segment records the item tying exactly with its u.q (the query
// itself when it is an item of P) in seg_self; a longer one lists such items
// of all its thresholds in self_col (ascending, each once, -1 after the last),
// each with its exact position in self_pos: its canonical score is its query's
// threshold, so it exceeds exactly the thresholds below that one.
__global__ void k_seg_prep(int64_t nseg, const int64_t *__restrict__ seg_start,
                           const int32_t *__restrict__ seg_len, const uint64_t *__restrict__ key_hi,
                           const int32_t *__restrict__ order, const double *__restrict__ th,
                           const int32_t *__restrict__ cq, const int32_t *__restrict__ qself,
                           int32_t *__restrict__ seg_user, int32_t *__restrict__ seg_self,
                           float2 *__restrict__ thr, double *__restrict__ ths,
                           uint32_t *__restrict__ hist,
                           int32_t *__restrict__ self_col, int32_t *__restrict__ self_pos) {
  int64_t sg = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (sg >= nseg) return;
  const int L = seg_len[sg];
  if (L == 0) return;   // a slot between the two ranges
  int64_t st0 = seg_start[sg];
  seg_user[sg] = (int32_t)key_hi[st0];
  seg_self[sg] = L == 1 ? qself[cq[order[st0]]] : -1;
  for (int i = 0; i < L; ++i) ths[st0 + i] = th[order[st0 + i]];
  for (int i = 0; i <= L; ++i) hist[2 * st0 + i] = 0;
  if (L == 1) {
    thr[sg] = make_float2(__double2float_rd(ths[st0]), __double2float_ru(ths[st0]));
    return;
  }
  int32_t *sc = self_col + st0, *sp = self_pos + st0;
  int ns = 0;
  for (int i = 0; i < L; ++i) {
    const int32_t c = qself[cq[order[st0 + i]]];
    if (c < 0) continue;
    int pos = i;
    while (pos > 0 && ths[st0 + pos - 1] == ths[st0 + i]) --pos;
    int at = ns;
    while (at > 0 && sc[at - 1] > c) --at;
    if (at > 0 && sc[at - 1] == c) continue;   // the same item for an equal query
    for (int j = ns; j > at; --j) {
      sc[j] = sc[j - 1];
      sp[j] = sp[j - 1];
    }
    sc[at] = c;
    sp[at] = pos;
    ++ns;
  }
  for (int j = ns; j < L; ++j) sc[j] = -1;
}

// hist[pos] counts items whose score exceeds exactly the first pos thresholds;
// after the suffix sum h[i] = #{p : s(u,p) > theta_{i-1}}.
__global__ void k_seg_suffix(int64_t nseg, const int64_t *__restrict__ seg_start,
                             const int32_t *__restrict__ seg_len, uint32_t *__restrict__ hist) {
  int64_t sg = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (sg >= nseg || seg_len[sg] == 0) return;
  uint32_t *h = hist + 2 * seg_start[sg];
  uint32_t run = 0;
  for (int i = seg_len[sg]; i >= 1; --i) {
    run += h[i];
    h[i] = run;
  }
}

// count of candidate order[st0 + i] = hist[2 st0 + i + 1] (see k_seg_suffix).
__global__ void k_scatter_counts(int64_t nseg, const int64_t *__restrict__ seg_start,
                                 const int32_t *__restrict__ seg_len,
                                 const int32_t *__restrict__ order,
                                 const uint32_t *__restrict__ hist, uint32_t *__restrict__ ccount) {
  int64_t sg = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (sg >= nseg) return;
  int L = seg_len[sg];
  if (L == 0) return;
  int64_t st0 = seg_start[sg];
  const uint32_t *h = hist + 2 * st0;
  for (int i = 0; i < L; ++i) ccount[order[st0 + i]] = h[i + 1];
}

// The deep count grid of an index (dg = 0: none).
struct DeepGrid {
  int dg;
  const BinFP *ybin;
  const uint32_t *DLO, *DHI;
};
inline DeepGrid deep_grid(const rkr_index *idx) {
  return DeepGrid{idx->dg, idx->ybin, idx->DLO, idx->DHI};
}

// Exact ranks from the tail lists.  A candidate (u, q) with u.q >= x_0(u)
// has rank 1 + #{p in list(u) : s(u,p) > u.q}, since every item scoring above
// x_0 is in the list.  Entries are grouped by exact-grid column: whole
// columns are counted from the column offsets, and the entries of the one or
// two columns within the screen bound of u.q are settled one by one, by their
// own bound, a compensated product, or canonically.  Candidates below x_0 (or with an overflowed list) are
// passed on, unchanged, in cu_fb for the recount screen; others get -1 there.
// 64 registers a thread (eight 128-thread blocks per SM): the kernel waits on
// scattered reads of each candidate's user data and list, so warps in flight matter.
__global__ void __launch_bounds__(128, 8) k_list_rank(int64_t count, const int32_t *__restrict__ cu,
                            const int32_t *__restrict__ cq, const float *__restrict__ cx,
                            const tc::RowBound *__restrict__ qrb, const float *__restrict__ U,
                            const float *__restrict__ unrm, const float *__restrict__ Q,
                            const float *__restrict__ Ps, const float *__restrict__ pnrm_s, int d,
                            const uint2 *__restrict__ xlist,
                            const int64_t *__restrict__ xloff, const uint32_t *__restrict__ xlcap,
                            const uint16_t *__restrict__ xcoff,
                            const uint32_t *__restrict__ xlcnt,
                            const float *__restrict__ xbmax, const tc::RowBound *__restrict__ rb3,
                            const tc::RowBound *__restrict__ ptile, int pbn, tc::Gacc gacc,
                            float gcan, const double *__restrict__ xg0,
                            const BinFP *__restrict__ xbin, int GX,
                            const double *__restrict__ ldx, const BinFP *__restrict__ lbin,
                            int G, const uint32_t *__restrict__ XLO,
                            const uint32_t *__restrict__ XHI, uint32_t mtop,
                            uint32_t *__restrict__ ccount, uint32_t *__restrict__ clb,
                            int32_t *__restrict__ cu_fb, const int32_t *__restrict__ qself,
                            DeepGrid deep, unsigned long long *__restrict__ stat) {
  int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= count) return;
  const int64_t u = cu[i];
  if (u < 0) {  // an unused slot or a pruned candidate: never selected
    cu_fb[i] = -1;
    ccount[i] = 0xffffffffu;
    clb[i] = 0xffffffffu;
    return;
  }
  const float *uu = U + u * d;
  const float *qq = Q + (int64_t)cq[i] * d;
  // u.q as an interval, tightened only where a comparison needs it: first the
  // candidate's screened score and its bound (no row is read), then the
  // compensated product, then the canonical value.  [flo, fhi] are its ends in
  // float, enough for every comparison with a screened entry; tlo, thi and theta
  // hold them in FP64 from the compensated product on.
  float flo = -INFINITY, fhi = INFINITY;
  double tlo = -INFINITY, thi = INFINITY;
  int state = 1;   // 0: screened interval, 1: compensated, 2: canonical
  auto compensate = [&]() {
    dot2_interval(uu, qq, d, tlo, thi);
    flo = __double2float_rd(tlo);
    fhi = __double2float_ru(thi);
    state = 1;
  };
  const float sx = cx ? cx[i] : __int_as_float(0x7fffffff);
  if (sx == sx) {
    const float b = tc::screen_bound_tc(rb3[u], qrb[cq[i]], gacc, gcan);
    flo = __fsub_rd(sx, b);
    fhi = __fadd_ru(sx, b);
    if (!(flo <= fhi)) {   // an infinite score within an infinite bound
      flo = -INFINITY;
      fhi = INFINITY;
    }
    state = 0;
  } else {
    compensate();
  }
  double theta = 0.0;
  auto tighten = [&]() {
    if (state == 0) {
      compensate();
    } else {
      theta = canon_dot(uu, qq, d);
      tlo = thi = theta;
      flo = __double2float_rd(theta);
      fhi = __double2float_ru(theta);
      state = 2;
      atomicAdd(&stat[4], 1ull);
    }
  };
  const uint32_t L = xlcnt[u];
  const bool full = L > xlcap[u];   // the list overflowed: not usable
  // u.q against x_0, whose nearest float is the list grid's origin
  const BinFP lb = lbin[u];
  bool under = fhi < nextafterf(lb.fmin32, -INFINITY);
  if (!under && flo < nextafterf(lb.fmin32, INFINITY)) {   // not decided in float
    const double x0 = xg0[u];
    if (state == 0) {
      tlo = (double)flo;
      thi = (double)fhi;
    }
    while (state < 2 && !full && tlo < x0 && thi >= x0) tighten();
    under = thi < x0;
  }
  if (full || under) {
    // bounds from the exact count table at the bins of both ends of u.q (below x_0:
    // before its first column)
    int jl = 0, jh = 0;
    if (!under) {
      const TightBins tb(xbin[u]);
      jl = tb.usable() ? tb.lo(flo, GX) : 0;
      jh = tb.usable() ? tb.hi(fhi, GX) : GX;
    }
    const int G2 = deep.dg;
    const bool below = G2 > 0 && under;
    int kl = 0, kh = G2;
    if (below) {
      const TightBins tb(deep.ybin[u]);
      if (tb.usable()) {
        kl = tb.lo(flo, G2);
        kh = tb.hi(fhi, G2);
      }
    }
    uint32_t ub = jl >= 1 ? XHI[u * GX + jl - 1] : mtop;
    uint32_t lb = jh < GX ? XLO[u * GX + jh] : 0u;
    if (below) {
      // below x_0: the deep grid's counts at y_{kl - 1} <= tlo and y_{kh} > thi
      if (kl >= 1) ub = min(ub, deep.DHI[u * G2 + kl - 1]);
      if (kh < G2) lb = max(lb, deep.DLO[u * G2 + kh]);
    }
    ccount[i] = ub;
    clb[i] = lb;
    cu_fb[i] = (int32_t)u;
    atomicAdd(&stat[0], 1ull);
    return;
  }
  cu_fb[i] = -1;
  // entries are grouped by column c = #{x_j <= v}: x_{c-1} <= v < x_c
  const uint2 *row = xlist + xloff[u];
  const uint16_t *co = xcoff + u * (G + 2);
  const float B = xbmax[u];
  // columns c >= chi have v >= x_{c-1} > u.q + B: every entry is above u.q;
  // columns c < clo have v < x_c <= u.q - B: no entry is above u.q (an upper and a
  // lower bound of these columns serve as well: the entries between are settled
  // one by one)
  int chi, clo;
  const TightBins tb(lb);
  if (tb.usable()) {
    chi = tb.hi(__fadd_ru(fhi, B), G) + 1;
    clo = tb.lo(__fsub_rd(flo, B), G);
  } else {
    const double g0 = xg0[u], dx = ldx[u];
    chi = exact_j((double)__fadd_ru(fhi, B), g0, dx, G) + 1;
    clo = exact_j((double)__fsub_rd(flo, B), g0, dx, G);
  }
  uint32_t above = L - (uint32_t)co[chi];
  const tc::RowBound ru = rb3[u];
  const int32_t self = qself[cq[i]];
  for (int e = co[clo]; e < (int)co[chi]; ++e) {
    const uint32_t p = row[e].x;
    if ((int32_t)p == self) continue;  // the query's own item: s(u,p) = u.q, not above
    const float v = __uint_as_float(row[e].y);
    const float b = tc::screen_bound_tc(ru, ptile[p / pbn], gacc, gcan);
    if (__fsub_rd(v, b) > fhi) { ++above; continue; }
    if (__fadd_ru(v, b) <= flo) continue;
    if (state == 0) {   // the screened interval of u.q cannot place it: compensate, look again
      tighten();
      --e;
      continue;
    }
    const float *pp = Ps + (int64_t)p * d;
    double slo, shi;
    dot2_interval(uu, pp, d, slo, shi);
    if (slo > thi) { ++above; continue; }
    if (shi <= tlo) continue;
    atomicAdd(&stat[1], 1ull);
    if (state < 2) tighten();   // the canonical u.q
    const double sc = canon_dot(uu, pp, d);
    if (sc > theta) ++above;
    // screen error of this pair against its canonical score: relative to the
    // bound (at most 1 for a sound bound) and to the norm bounds ||u|| ||p||
    const double er = fabs((double)v - sc);
    const float ratio = (float)(er / (double)b);
    const float rel = (float)(er / ((double)unrm[u] * (double)pnrm_s[p]));
    atomicMax(&stat[2], (unsigned long long)__float_as_uint(ratio));
    atomicMax(&stat[3], (unsigned long long)__float_as_uint(rel));
  }
  ccount[i] = above;
  clb[i] = above;
}

// Threads of the per-query filters.  One CTA walks a query's candidates, up to a
// million, and waits for its loads: 1,024 threads with eight in flight where a query
// has thousands (67k each of 1,024 queries: k_recount_filter 12.3 -> 4.8 ms; 9k each
// of 512: 2.1 -> 0.8 ms, against 512 threads with four).  Many queries with few each
// fill the SMs by themselves (1.6k each of 10,000: 1,024 threads 0.85 ms, 512 0.50).
constexpr int kFilterThreads = 1024;
static int filter_threads(int64_t candidates, int queries) {
  return candidates >= (int64_t)4096 * queries ? kFilterThreads : kFilterThreads / 2;
}

// k-th smallest of the counts cc[0 .. cnt) (each at most top, or ~0), walking only
// the bytes such counts have.
__device__ __forceinline__ uint64_t block_kth_count(const uint32_t *cc, int64_t cnt, uint64_t k,
                                                    uint64_t top, uint32_t *hist, uint64_t *bc) {
  const int bits = count_bits(top);
  const uint64_t r = block_kth<8>(cnt, k, bits,
                               [&](int64_t i, uint64_t &key) {
                                 key = count_key(cc[i], bits);
                                 return true;
                               },
                               hist, bc);
  return r == ((uint64_t)1 << bits) - 1 ? 0xffffffffull : r;
}

// Per query: cap = k-th smallest of (exact count, or upper bound for candidates
// still to be recounted).  A candidate whose lower bound exceeds the cap cannot
// be among the k smallest ranks: it is dropped from the recount and given the
// largest key.
__global__ void __launch_bounds__(kFilterThreads)
    k_recount_filter(int qa, const int64_t *__restrict__ qoff, const uint32_t *__restrict__ qcount,
                     const int32_t *__restrict__ kq, uint32_t *__restrict__ ccount,
                     const uint32_t *__restrict__ clb, int32_t *__restrict__ cu_fb,
                     uint32_t mtop) {
  __shared__ __align__(16) uint32_t hist[256];
  __shared__ uint64_t bc[2];
  const int q = qa + blockIdx.x;
  const int64_t base = qoff[q] - qoff[qa];
  const int64_t cnt = qcount[q];
  const int k = kq[q];
  if (cnt < k) return;
  uint32_t *cc = ccount + base;
  const uint32_t *lb = clb + base;
  int32_t *fb = cu_fb + base;
  const uint64_t cap = block_kth_count(cc, cnt, (uint64_t)k, mtop, hist, bc);
  for (int64_t i0 = threadIdx.x; i0 < cnt; i0 += 8 * (int64_t)blockDim.x) {
    int32_t f[8];
    uint32_t b[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) {   // loads in flight together
      const int64_t i = i0 + j * (int64_t)blockDim.x;
      f[j] = i < cnt ? fb[i] : -1;
      b[j] = i < cnt ? lb[i] : 0u;
    }
#pragma unroll
    for (int j = 0; j < 8; ++j)
      if (f[j] >= 0 && (uint64_t)b[j] > cap) {
        const int64_t i = i0 + j * (int64_t)blockDim.x;
        fb[i] = -1;
        cc[i] = 0xffffffffu;
      }
  }
}

__global__ void k_count_valid(int64_t n, const int32_t *__restrict__ v,
                              unsigned long long *__restrict__ out) {
  int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  unsigned long long c = (i < n && v[i] >= 0) ? 1ull : 0ull;
  c = __reduce_add_sync(0xffffffffu, (unsigned)c);
  if ((threadIdx.x & 31) == 0 && c) atomicAdd(out, c);
}

// Early termination over the norm-sorted items (tuning rc_prefix).  A query
// takes part when at least prefix_min_rows(k) of its candidates still need a
// recount; those candidates are copied to cu_pre for the prefix pass.
__host__ __device__ inline int64_t prefix_pick_rows(int k) { return k * 8 > 256 ? k * 8 : 256; }
__host__ __device__ inline int64_t prefix_min_rows(int k) { return 8 * prefix_pick_rows(k); }

__global__ void __launch_bounds__(256)
    k_prefix_split(int qa, const int64_t *__restrict__ qoff, const uint32_t *__restrict__ qcount,
                   const int32_t *__restrict__ kq, const int32_t *__restrict__ cu_fb,
                   int32_t *__restrict__ cu_pre, unsigned long long *__restrict__ npre) {
  __shared__ unsigned long long acc;
  const int q = qa + blockIdx.x;
  const int64_t base = qoff[q] - qoff[qa];
  const int64_t cnt = qcount[q];
  const int32_t *fb = cu_fb + base;
  const int64_t nr = block_count(cnt, [&](int64_t i) { return fb[i] >= 0; }, &acc);
  if (nr < prefix_min_rows(kq[q])) return;
  for (int64_t i = threadIdx.x; i < cnt; i += blockDim.x) cu_pre[base + i] = fb[i];
  if (threadIdx.x == 0) atomicAdd(npre, (unsigned long long)nr);
}

// Per query of the prefix pass: every prefix row's lower bound takes its certain
// count over the prefix (a subset of P); the prefix_pick_rows(k) rows with the
// smallest possible prefix counts (ties included) stay in cu_fb for a recount
// over all of P, the others are parked in cu_park until the cap is known.
__global__ void __launch_bounds__(kFilterThreads)
    k_prefix_pick(int qa, const int64_t *__restrict__ qoff, const uint32_t *__restrict__ qcount,
                  const int32_t *__restrict__ kq, const int32_t *__restrict__ cu_pre,
                  const uint32_t *__restrict__ hi1, const uint32_t *__restrict__ lo1,
                  uint32_t *__restrict__ clb, int32_t *__restrict__ cu_fb,
                  int32_t *__restrict__ cu_park) {
  __shared__ __align__(16) uint32_t hist[256];
  __shared__ uint64_t bc[2];
  __shared__ unsigned long long acc;
  const int q = qa + blockIdx.x;
  const int64_t base = qoff[q] - qoff[qa];
  const int64_t cnt = qcount[q];
  const int32_t *pre = cu_pre + base;
  const int64_t np = block_count(cnt, [&](int64_t i) { return pre[i] >= 0; }, &acc);
  const uint64_t k2 = (uint64_t)prefix_pick_rows(kq[q]);
  if (np <= (int64_t)k2) return;
  const uint32_t *h = hi1 + base, *l = lo1 + base;
  const uint64_t T = block_kth(cnt, k2, 32,
                               [&](int64_t i, uint64_t &key) {
                                 key = h[i];
                                 return pre[i] >= 0;
                               },
                               hist, bc);
  for (int64_t i = threadIdx.x; i < cnt; i += blockDim.x) {
    if (pre[i] < 0) continue;
    clb[base + i] = max(clb[base + i], l[i]);
    if ((uint64_t)h[i] > T) {
      cu_park[base + i] = cu_fb[base + i];
      cu_fb[base + i] = -1;
    }
  }
}

// Parked rows that the cap did not drop go back to the recount.
__global__ void k_prefix_unpark(int64_t n, const int32_t *__restrict__ cu_park,
                                int32_t *__restrict__ cu_fb) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i < n && cu_park[i] >= 0) cu_fb[i] = cu_park[i];
}

// One CTA per query: the k smallest (rank, index) among its candidates.
__global__ void __launch_bounds__(kSelThreadsFew)
    k_select_exact(int qa, const int64_t *__restrict__ qoff, const uint32_t *__restrict__ qcount,
                   const int32_t *__restrict__ cuid,
                   const uint32_t *__restrict__ ccount, const int32_t *__restrict__ kq,
                   const int64_t *__restrict__ out_off, int32_t *__restrict__ out_users,
                   int32_t *__restrict__ out_ranks, int *__restrict__ err, uint32_t mtop,
                   int ubits) {
  extern __shared__ unsigned char sbuf[];
  SortEnt *ent = (SortEnt *)sbuf;
  __shared__ __align__(16) uint32_t hist[256];
  __shared__ uint64_t bc[2];
  __shared__ int gcount;
  const int q = qa + blockIdx.x;
  const int64_t base = qoff[q] - qoff[qa];
  const int64_t cnt = qcount[q];
  const int k = kq[q];
  if (cnt < k) {
    if (threadIdx.x == 0) atomicExch(err, 1);
    return;
  }
  const int32_t *uid = cuid + base;
  const uint32_t *cc = ccount + base;
  // (count, user) packed into the bytes they need: mtop bounds the counts (~0 marks
  // a dropped candidate), ubits (a multiple of 8) the users
  const int cbits = count_bits(mtop);
  auto key_of = [&](int64_t i) {
    const uint32_t u = uid[i] < 0 ? 0u : (uint32_t)uid[i];   // (dropped: behind every count)
    return (count_key(cc[i], cbits) << ubits) | u;
  };
  uint32_t upto;
  const uint64_t last = block_kth_cut(cnt, (uint64_t)k, cbits + ubits,
                                      [&](int64_t i, uint64_t &key) {
                                        key = key_of(i);
                                        return true;
                                      },
                                      hist, bc, sort_room(k), upto);
  if (threadIdx.x == 0) gcount = 0;
  __syncthreads();
  for (int64_t i = threadIdx.x; i < cnt; i += blockDim.x) {
    if (key_of(i) <= last) {
      int pos = atomicAdd(&gcount, 1);
      if (pos < kMaxK) {
        ent[pos].k1 = ((uint64_t)cc[i] << 32) | (uint32_t)uid[i];
        ent[pos].k2 = 0;
        ent[pos].idx = (int32_t)i;
      }
    }
  }
  __syncthreads();
  int got = min(gcount, kMaxK);
  block_sort(ent, got);
  const int64_t obase = out_off[q];
  for (int r = threadIdx.x; r < got && r < k; r += blockDim.x) {
    out_users[obase + r] = (int32_t)(ent[r].k1 & 0xffffffffu);
    out_ranks[obase + r] = (int32_t)(ent[r].k1 >> 32) + 1;
  }
}

// ------------------------------------------------------------------- host

// ------------------------------------------------------------ skim list

// Entry e of region blockIdx.y (thread index within the region's count).
__device__ __forceinline__ bool list_entry(const SkimList &L, int64_t &e) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const uint32_t c = L.cnt[blockIdx.y];
  if (i >= (int64_t)(c < L.rcap ? c : L.rcap)) return false;
  e = (int64_t)blockIdx.y * L.rcap + i;
  return true;
}

// Pass 1 on the list: bin interval of each entry's u.q from its screened score
// and the pair's own bound, the levels of its upper and lower rank bounds
// (histograms per query), and both kept for the later passes.
__global__ void k_list_levels(SkimList L, const tc::RowBound *__restrict__ urb,
                              const tc::RowBound *__restrict__ qrb, tc::Gacc gacc, float gcan,
                              const BinFP *__restrict__ bf, const double *__restrict__ fmin,
                              int tau, const int16_t *__restrict__ JU,
                              const int16_t *__restrict__ JL, uint32_t *__restrict__ hist_up,
                              uint32_t *__restrict__ hist_lo, uint32_t *__restrict__ jj,
                              uint32_t *__restrict__ lv, const uint32_t *__restrict__ member,
                              int64_t mwords) {
  int64_t e;
  if (!list_entry(L, e)) return;
  const int64_t u = L.u[e];
  const int q = L.q[e];
  if (!in_subset(member, mwords, q, u)) {  // outside the query's subset: never counted
    jj[e] = 0;
    lv[e] = 0xffffu;
    return;
  }
  const float x = L.x[e];
  const float b = tc::screen_bound_tc(urb[u], qrb[q], gacc, gcan);
  int jlo, jhi;
  bin_interval(bf[u], fmin[u], tau, __fsub_rd(x, b), __fadd_ru(x, b), jlo, jhi);
  const int16_t *ju = JU + u * kMaxLevels, *jl = JL + u * kMaxLevels;
  int lu = 0, ll = 0;
#pragma unroll
  for (int step = 16; step > 0; step >>= 1) {
    if (ju[lu + step - 1] > jlo) lu += step;
    if (jl[ll + step - 1] > jhi) ll += step;
  }
  atomicAdd(&hist_up[(int64_t)q * 32 + lu], 1u);
  atomicAdd(&hist_lo[(int64_t)q * 32 + ll], 1u);
  jj[e] = (uint32_t)jlo | ((uint32_t)jhi << 16);
  lv[e] = (uint32_t)lu | ((uint32_t)ll << 8);
}

// Pass 3 on the list: entries whose upper bound lies exactly at their query's
// level L* add that bound to the query's fine histogram of the level.
__global__ void k_list_fine(SkimList L, const uint32_t *__restrict__ jj,
                            const uint32_t *__restrict__ lv, const int32_t *__restrict__ lstar,
                            int lskip, const uint32_t *__restrict__ thi, int tau, uint32_t top,
                            uint32_t scale, uint32_t *__restrict__ fine) {
  int64_t e;
  if (!list_entry(L, e)) return;
  const int q = L.q[e];
  const int Lq = lstar[q];
  if (Lq > lskip || (int)(lv[e] & 0xff) != Lq) return;
  const int64_t u = L.u[e];
  const int jlo = (int)(jj[e] & 0xffff);
  const uint64_t v = jlo >= 1 ? thi[u * tau + jlo - 1] : top;
  const uint64_t hi = level_bound(Lq, scale);
  const uint64_t base = Lq == 0 ? 0 : level_bound(Lq - 1, scale) + 1;
  const uint64_t width = (hi - base + 1024) / 1024;
  uint64_t bkt = v >= base ? (v - base) / width : 0;
  if (bkt >= 1024) bkt = 1023;
  atomicAdd(&fine[(int64_t)q * 1024 + bkt], 1u);
}

// Pass 2 on the list: entries of queries [qa, qb) whose lower bound may reach
// the query's refined cap, appended to the query's candidate segment with their
// screened score (its bound settles most later decisions about u.q).
__global__ void k_list_emit(SkimList L, const uint32_t *__restrict__ jj,
                            const uint32_t *__restrict__ lv, int qa, int qb,
                            const int32_t *__restrict__ lstar, int lskip,
                            const uint32_t *__restrict__ cap, const uint32_t *__restrict__ tlo,
                            int tau, const int64_t *__restrict__ qoff,
                            uint32_t *__restrict__ qcursor, int32_t *__restrict__ cand_u,
                            int32_t *__restrict__ cand_q, float *__restrict__ cand_x,
                            int *__restrict__ ovf) {
  int64_t e;
  if (!list_entry(L, e)) return;
  const int q = L.q[e];
  if (q < qa || q >= qb) return;
  const int Lq = lstar[q];
  if (Lq > lskip || (int)((lv[e] >> 8) & 0xff) > Lq) return;
  const int64_t u = L.u[e];
  const int jhi = (int)(jj[e] >> 16);
  const uint32_t lb = jhi < tau ? tlo[u * tau + jhi] : 0u;
  if (lb > cap[q]) return;
  const uint32_t pos = atomicAdd(&qcursor[q], 1u);
  const int64_t at = qoff[q] + pos;
  if (at >= qoff[q + 1]) {
    atomicExch(ovf, 1);
    return;
  }
  cand_u[at] = (int32_t)u;
  cand_q[at] = q;
  cand_x[at] = L.x[e];
}

// Shared front half: passes 1 and 3 and the cutoffs; per-query candidate counts.
// Pairs whose lower bound lies above the skip level are left out by a single
// compare of the screened score; queries whose cutoff lies above it ("deep")
// are gathered and screened again in full by launches of their own.
struct Plan {
  std::vector<int64_t> ncand;
  std::vector<int32_t> lstar;
  int lskip = 1 << 30;          // skip level (no skipping: every level)
  DevBuf bxs;
  float *xs = nullptr;          // per-user skip scores
  std::vector<int32_t> deep;    // deep queries, ascending
  DevBuf bdeep, bdhi, bdlo, bdr1, bdr3;
  int32_t *deep_d = nullptr;
  TcSide dside;                 // their bf16 rows (views of the buffers above)
  bool listed = false;          // passes 1-3 of the other queries run on the skim list
  SkimList list{};
  uint32_t maxcnt = 0;          // largest region count (launch width of list kernels)
  DevBuf blu, blq, blx, blc, bjj, blv;
  uint32_t *jj = nullptr, *lv = nullptr;
};

static rkr_status check_flag(int *flag_d, const char *what, cudaStream_t st);

// Capacity of the skim list: entries of every region together.
static int64_t skim_capacity(int64_t n, int64_t nq) {
  int64_t want = n * nq / 16;
  return std::max<int64_t>((int64_t)1 << 20, std::min<int64_t>(want, (int64_t)1 << 29));
}

static dim3 list_grid(const Plan &plan) {
  return dim3((unsigned)std::max<uint32_t>(1, (plan.maxcnt + 255) / 256),
              (unsigned)plan.list.regions);
}

// Skim screen of all queries into plan.list; plan.listed stays false when the
// list cannot be allocated or a region overflowed (the passes then screen again).
static rkr_status skim_queries(const rkr_index *idx, const QueryCommon &qc, int nq, Plan &plan,
                               int *flag, cudaStream_t st) {
  const int regions = skim_regions(idx->n, nq);
  const int64_t cap = skim_capacity(idx->n, nq);
  SkimList &L = plan.list;
  L.regions = regions;
  L.rcap = cap / regions;
  const size_t ent = (size_t)L.rcap * regions;
  auto try_alloc = [&](DevBuf &b, auto **p, size_t count) -> bool {
    cudaError_t e = pool_malloc_async((void **)p, count * sizeof(**p), st);
    if (e != cudaSuccess) {
      cudaGetLastError();
      return false;
    }
    b.p = (void *)*p;
    b.st = st;
    return true;
  };
  if (!try_alloc(plan.blu, &L.u, ent) || !try_alloc(plan.blq, &L.q, ent) ||
      !try_alloc(plan.blx, &L.x, ent) || !try_alloc(plan.blc, &L.cnt, regions + 1) ||
      !try_alloc(plan.bjj, &plan.jj, ent) || !try_alloc(plan.blv, &plan.lv, ent))
    return RKR_OK;
  RKR_CUDA(cudaMemsetAsync(L.cnt, 0, sizeof(uint32_t) * regions, st));
  RKR_TRY(tc_skim(idx, idx->Ut, qc.Qt, plan.xs, L, flag, st));
  std::vector<uint32_t> cnt(regions + 1);
  // (the screen's error word stands behind the counts: one transfer)
  RKR_CUDA(cudaMemcpyAsync(L.cnt + regions, flag, sizeof(int), cudaMemcpyDeviceToDevice, st));
  RKR_CUDA(cudaMemcpyAsync(cnt.data(), L.cnt, sizeof(uint32_t) * (regions + 1),
                           cudaMemcpyDeviceToHost, st));
  RKR_CUDA(cudaStreamSynchronize(st));
  if (cnt[regions]) return fail(RKR_ETIMEOUT, "skim screen: screen kernel wait timed out (%d)",
                                (int)cnt[regions]);
  cnt.resize(regions);
  uint32_t mx = 0;
  for (uint32_t c : cnt) {
    if ((int64_t)c > L.rcap) return RKR_OK;  // overflow: not listed
    mx = std::max(mx, c);
  }
  plan.maxcnt = mx;
  plan.listed = true;
  return RKR_OK;
}

// Skip level: the smallest level whose ranks reach m / 128.
static int skip_level(const rkr_index *idx) {
  const char *env = getenv("RKR_SKIP_LEVEL");
  if (env && *env) return atoi(env);
  const int tl = tuning().skip_level;
  if (tl > 0) return tl;
  int64_t r = idx->m / 128;
  int L = 0;
  while (L < 31 && (((int64_t)1 << L) - 1) < r) ++L;
  return L;
}

// Grid, bin parameters, level tables and bound tables of one path.
struct Grid {
  const BinFP *bf;
  const double *fmin;
  int tau;
  const int16_t *JU, *JL;
  int nlev;
  const uint32_t *thi, *tlo;
  uint32_t top, scale;
};

constexpr int kThetaSplit = 1;  // u.q screened with the split (three-term) product

static rkr_status check_flag(int *flag_d, const char *what, cudaStream_t st) {
  int h = 0;
  RKR_CUDA(cudaMemcpyAsync(&h, flag_d, sizeof(int), cudaMemcpyDeviceToHost, st));
  RKR_CUDA(cudaStreamSynchronize(st));
  if (h) return fail(RKR_ETIMEOUT, "%s: screen kernel wait timed out (%d)", what, h);
  return RKR_OK;
}

static ThetaArgs theta_args(const Grid &g, int qa, const QueryCommon &qc) {
  ThetaArgs a{};
  a.qa = qa;
  a.lskip = 1 << 30;
  a.member = qc.member;
  a.mwords = qc.mwords;
  a.binfp = g.bf;
  a.fmin = g.fmin;
  a.tau = g.tau;
  a.JU = g.JU;
  a.JL = g.JL;
  a.thi = g.thi;
  a.tlo = g.tlo;
  a.top = g.top;
  a.scale = g.scale;
  return a;
}

// Bytes of the plan's per-query results: int64 candidate counts, int32 levels, then
// the screens' error word.
static size_t plan_bytes(int nq) { return (sizeof(int64_t) + sizeof(int32_t)) * nq + sizeof(int); }

// Passes 1 and 3: per-query cutoff level, refined cap, and candidate-count bounds.
static rkr_status screen_plan(const rkr_index *idx, const QueryCommon &qc, int nq,
                              const Grid &g, cudaStream_t st, int32_t *lstar_d, uint32_t *cap_d,
                              int64_t *ncand_d, Plan &plan) {
  DevBuf bh, bf, bb, bfi;
  uint32_t *hist, *fine;
  uint64_t *below;
  int *flag;
  RKR_TRY(tmp_alloc(bh, &hist, (size_t)nq * 64, st));
  RKR_TRY(tmp_alloc(bfi, &fine, (size_t)nq * 1024, st));
  RKR_TRY(tmp_alloc(bb, &below, nq, st));
  RKR_TRY(tmp_alloc(bf, &flag, 1, st));
  RKR_CUDA(cudaMemsetAsync(hist, 0, sizeof(uint32_t) * (size_t)nq * 64, st));
  RKR_CUDA(cudaMemsetAsync(fine, 0, sizeof(uint32_t) * (size_t)nq * 1024, st));
  RKR_CUDA(cudaMemsetAsync(flag, 0, sizeof(int), st));
  const int LS = skip_level(idx);
  const bool skip = LS >= 0 && LS < g.nlev - 1;
  if (skip) {
    RKR_TRY(tmp_alloc(plan.bxs, &plan.xs, idx->n, st));
    k_skip_scores<<<(unsigned)((idx->n + 255) / 256), 256, 0, st>>>(idx->n, g.bf, g.JL, LS,
                                                                     plan.xs);
    note_launch();
    RKR_CUDA(cudaGetLastError());
    plan.lskip = LS;
  }
  ThetaArgs a = theta_args(g, 0, qc);
  a.nq_all = nq;
  a.hist = hist;
  a.xs = plan.xs;
  a.lskip = plan.lskip;
  if (skip) RKR_TRY(skim_queries(idx, qc, nq, plan, flag, st));
  if (plan.listed) {
    if (plan.maxcnt > 0) {
      {
        const int prof_slot = prof_begin("k_list_levels", st);
        k_list_levels<<<list_grid(plan), 256, 0, st>>>(
            plan.list, idx->Ut.rb3, qc.Qt.rb3, tc_gacc(idx->Ut.kp, 1), tc_gcan(idx->d), g.bf,
            g.fmin, g.tau, g.JU, g.JL, hist, hist + (size_t)nq * 32, plan.jj, plan.lv, qc.member,
          qc.mwords);
        prof_end(prof_slot, st, 0.0);
      }
      note_launch();
      RKR_CUDA(cudaGetLastError());
    }
  } else {
    RKR_TRY(tc_theta_pass(1, idx, idx->Ut, qc.Qt, a, kThetaSplit, flag, st));
  }
  k_cutoff<<<(nq + 127) / 128, 128, 0, st>>>(nq, hist, hist + (size_t)nq * 32, qc.kq_d, g.nlev,
                                             skip ? LS : 31, lstar_d, below, ncand_d);
  note_launch();
  RKR_CUDA(cudaGetLastError());
  ThetaArgs ad = a;  // deep queries: own rows, every pair screened
  ad.xs = nullptr;
  ad.lskip = 1 << 30;
  if (skip) {
    std::vector<int32_t> ls(nq);
    RKR_CUDA(cudaMemcpyAsync(ls.data(), lstar_d, sizeof(int32_t) * nq, cudaMemcpyDeviceToHost,
                             st));
    RKR_CUDA(cudaStreamSynchronize(st));
    for (int q = 0; q < nq; ++q)
      if (ls[q] == kDeep) plan.deep.push_back(q);
  }
  const int nd = (int)plan.deep.size();
  if (nd > 0) {
    const int kp = qc.Qt.kp, ld = qc.Qt.ld();
    TcSide &D = plan.dside;
    RKR_TRY(tmp_alloc(plan.bdeep, &plan.deep_d, nd, st));
    RKR_TRY(tmp_alloc(plan.bdhi, &D.hi, (size_t)nd * ld, st));
    RKR_TRY(tmp_alloc(plan.bdlo, &D.lo, (size_t)nd * ld, st));
    RKR_TRY(tmp_alloc(plan.bdr1, &D.rb1, nd, st));
    RKR_TRY(tmp_alloc(plan.bdr3, &D.rb3, nd, st));
    D.rows = nd;
    D.d = qc.Qt.d;
    D.kp = kp;
    D.pitch = qc.Qt.pitch;
    D.owned = false;
    RKR_CUDA(cudaMemcpyAsync(plan.deep_d, plan.deep.data(), sizeof(int32_t) * nd,
                             cudaMemcpyHostToDevice, st));
    {
      const int prof_slot = prof_begin("k_gather_qrows", st);
      k_gather_qrows<<<nd, 128, 0, st>>>(nd, plan.deep_d, kp, ld, qc.Qt.hi, qc.Qt.lo, qc.Qt.rb1,
                                         qc.Qt.rb3, D.hi, D.lo, D.rb1, D.rb3, hist, nq);
      prof_end(prof_slot, st, 0.0);
    }
    note_launch();
    RKR_CUDA(cudaGetLastError());
    ad.qmap = plan.deep_d;
    RKR_TRY(tc_theta_pass(1, idx, idx->Ut, D, ad, kThetaSplit, flag, st));
    k_cutoff<<<(nq + 127) / 128, 128, 0, st>>>(nq, hist, hist + (size_t)nq * 32, qc.kq_d,
                                               g.nlev, 31, lstar_d, below, ncand_d);
    note_launch();
    RKR_CUDA(cudaGetLastError());
  }
  a.hist = nullptr;
  a.lstar = lstar_d;
  a.fine = fine;
  if (plan.listed) {
    if (plan.maxcnt > 0) {
      {
        const int prof_slot = prof_begin("k_list_fine", st);
        k_list_fine<<<list_grid(plan), 256, 0, st>>>(plan.list, plan.jj, plan.lv, lstar_d,
                                                     plan.lskip, g.thi, g.tau, g.top, g.scale,
                                                     fine);
        prof_end(prof_slot, st, 0.0);
      }
      note_launch();
      RKR_CUDA(cudaGetLastError());
    }
  } else {
    RKR_TRY(tc_theta_pass(3, idx, idx->Ut, qc.Qt, a, kThetaSplit, flag, st));
  }
  if (nd > 0) {
    ad.hist = nullptr;
    ad.lstar = lstar_d;
    ad.fine = fine;
    RKR_TRY(tc_theta_pass(3, idx, idx->Ut, plan.dside, ad, kThetaSplit, flag, st));
  }
  k_cutoff_fine<<<(nq + 127) / 128, 128, 0, st>>>(nq, fine, below, lstar_d, qc.kq_d, g.scale,
                                                  cap_d);
  note_launch();
  RKR_CUDA(cudaGetLastError());
  // candidate counts, cutoff levels and the error word lie behind one another
  plan.ncand.resize(nq);
  plan.lstar.resize(nq);
  std::vector<char> h(plan_bytes(nq));
  RKR_CUDA(cudaMemcpyAsync((char *)ncand_d + h.size() - sizeof(int), flag, sizeof(int),
                           cudaMemcpyDeviceToDevice, st));
  RKR_CUDA(cudaMemcpyAsync(h.data(), ncand_d, h.size(), cudaMemcpyDeviceToHost, st));
  RKR_CUDA(cudaStreamSynchronize(st));
  memcpy(plan.ncand.data(), h.data(), sizeof(int64_t) * nq);
  memcpy(plan.lstar.data(), h.data() + sizeof(int64_t) * nq, sizeof(int32_t) * nq);
  int err = 0;
  memcpy(&err, h.data() + h.size() - sizeof(int), sizeof(int));
  if (err) return fail(RKR_ETIMEOUT, "theta passes 1 and 3: screen kernel wait timed out (%d)", err);
  return RKR_OK;
}

// Error words and counters of one query call on the device, read once at its end
// (zeroed at its start).  Every write of a failed screen stays within its buffers.
struct CallWords {
  int screen_err, overflow, select_err, pad;
  unsigned long long nfp64, candidates, ties[2];
};
static rkr_status words_alloc(DevBuf &b, CallWords **w, cudaStream_t st) {
  RKR_TRY(tmp_alloc(b, w, 1, st));
  RKR_CUDA(cudaMemsetAsync(*w, 0, sizeof(CallWords), st));
  return RKR_OK;
}
// Reads them (waiting for the stream) and turns errors into a status.
static rkr_status words_check(const CallWords *w, CallWords &h, cudaStream_t st) {
  RKR_CUDA(cudaMemcpyAsync(&h, w, sizeof(h), cudaMemcpyDeviceToHost, st));
  RKR_CUDA(cudaStreamSynchronize(st));
  if (h.screen_err)
    return fail(RKR_ETIMEOUT, "theta pass 2: screen kernel wait timed out (%d)", h.screen_err);
  if (h.overflow) return fail(RKR_EINTERNAL, "candidate segment overflow in theta pass 2");
  if (h.select_err) return fail(RKR_EINTERNAL, "fewer than k candidates for a query");
  return RKR_OK;
}

// Sums the candidates of queries [qa, qb).  A cursor that ran past its segment
// (reported as overflow) goes back to the segment's end: what follows reads no further.
__global__ void k_close_segments(int qa, int qb, const int64_t *__restrict__ qoff,
                                 uint32_t *__restrict__ cursor,
                                 unsigned long long *__restrict__ sum) {
  unsigned long long s = 0;
  for (int q = qa + blockIdx.x * blockDim.x + threadIdx.x; q < qb; q += gridDim.x * blockDim.x) {
    const int64_t room = qoff[q + 1] - qoff[q];
    if ((int64_t)cursor[q] > room) cursor[q] = (uint32_t)room;
    s += cursor[q];
  }
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if ((threadIdx.x & 31) == 0 && s) atomicAdd(sum, s);
}

// Pass 2: candidates of queries [qa, qb) appended to per-query segments.  Nothing is
// waited for: errors stand in *words.  cand_x gets the screened scores of listed
// candidates and, with screen_x, those of the screen's own candidates too.
static rkr_status emit_candidates(const rkr_index *idx, const QueryCommon &qc, int qa, int qb,
                                  const Grid &g, const Plan &plan, const int32_t *lstar_d,
                                  const uint32_t *cap_d, const int64_t *qoff_d, uint32_t *cursor_d,
                                  int32_t *cand_u, int32_t *cand_q, float *cand_x,
                                  bool screen_x, CallWords *words, cudaStream_t st) {
  TcSide sub = qc.Qt;
  sub.owned = false;
  sub.rows = qb - qa;
  sub.hi = qc.Qt.hi + (size_t)qa * qc.Qt.ld();
  sub.lo = qc.Qt.lo + (size_t)qa * qc.Qt.ld();
  if (qc.Qt.cat) sub.cat = qc.Qt.cat + (size_t)qa * tc_pitch(3 * qc.Qt.kp);
  sub.rb1 = qc.Qt.rb1 + qa;
  sub.rb3 = qc.Qt.rb3 + qa;
  int *flag = &words->screen_err;
  ThetaArgs a = theta_args(g, qa, qc);
  a.nq_all = qc.Qt.rows;
  a.ovf = &words->overflow;
  a.lstar = lstar_d;
  a.cap = cap_d;
  a.qoff = qoff_d;
  a.qcursor = cursor_d;
  a.cand_u = cand_u;
  a.cand_q = cand_q;
  a.cand_x = screen_x ? cand_x : nullptr;
  a.xs = plan.xs;
  a.lskip = plan.lskip;
  if (plan.listed) {
    if (plan.maxcnt > 0) {
      {
        const int prof_slot = prof_begin("k_list_emit", st);
        k_list_emit<<<list_grid(plan), 256, 0, st>>>(plan.list, plan.jj, plan.lv, qa, qb, lstar_d,
                                                     plan.lskip, cap_d, g.tlo, g.tau, qoff_d,
                                                     cursor_d, cand_u, cand_q, cand_x,
                                                     &words->overflow);
        prof_end(prof_slot, st, 0.0);
      }
      note_launch();
      RKR_CUDA(cudaGetLastError());
    }
  } else {
    RKR_TRY(tc_theta_pass(2, idx, idx->Ut, sub, a, kThetaSplit, flag, st));
  }
  // deep queries of [qa, qb): a contiguous slice of the gathered rows
  const int da = (int)(std::lower_bound(plan.deep.begin(), plan.deep.end(), qa) - plan.deep.begin());
  const int db = (int)(std::lower_bound(plan.deep.begin(), plan.deep.end(), qb) - plan.deep.begin());
  if (db > da) {
    TcSide ds = plan.dside;
    ds.owned = false;
    ds.rows = db - da;
    ds.hi = plan.dside.hi + (size_t)da * ds.ld();
    ds.lo = plan.dside.lo + (size_t)da * ds.ld();
    ds.rb1 = plan.dside.rb1 + da;
    ds.rb3 = plan.dside.rb3 + da;
    ThetaArgs ad = a;
    ad.qmap = plan.deep_d + da;
    ad.xs = nullptr;
    ad.lskip = 1 << 30;
    RKR_TRY(tc_theta_pass(2, idx, idx->Ut, ds, ad, kThetaSplit, flag, st));
  }
  k_close_segments<<<std::min((qb - qa + 255) / 256, 64), 256, 0, st>>>(qa, qb, qoff_d, cursor_d,
                                                                        &words->candidates);
  note_launch();
  RKR_CUDA(cudaGetLastError());
  return RKR_OK;
}

// Group queries into chunks whose candidate total stays within budget.
static std::vector<std::pair<int, int>> chunk_queries(const std::vector<int64_t> &ncand,
                                                      int64_t budget) {
  std::vector<std::pair<int, int>> out;
  int nq = (int)ncand.size();
  int a = 0;
  while (a < nq) {
    int64_t tot = 0;
    int b = a;
    while (b < nq && (b == a || tot + ncand[b] <= budget)) tot += ncand[b++];
    out.push_back({a, b});
    a = b;
  }
  return out;
}

static int64_t candidate_budget() { return (int64_t)1 << tuning().cand_budget_log2; }

// The valid candidates (cu >= 0) one behind another, each with its index in oi; their
// order is that of the atomic cursor.
__global__ void k_compact(int64_t n, const int32_t *__restrict__ cu, const int32_t *__restrict__ cq,
                          unsigned long long *__restrict__ cursor, int32_t *__restrict__ ou,
                          int32_t *__restrict__ oq, int32_t *__restrict__ oi) {
  int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= n || cu[i] < 0) return;
  unsigned long long p = atomicAdd(cursor, 1ull);
  ou[p] = cu[i];
  oq[p] = cq[i];
  oi[p] = (int32_t)i;
}

__global__ void k_scatter_back(int64_t n, const int32_t *__restrict__ oi,
                               const uint32_t *__restrict__ c2, uint32_t *__restrict__ ccount) {
  int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= n) return;
  ccount[oi[i]] = c2[i];
}

// Rows of a recount with one threshold each: the row's threshold and the item tying
// exactly with it.  With cx (the screened scores of all candidates, by their index
// ci) a row whose candidate has a screened score takes the interval [score - bound,
// score + bound] holding u.q as its threshold, so no row of U or Q is read (unless the
// score and its bound are infinite).  The others take the canonical u.q rounded both
// ways (ths, when wanted, gets the value itself).  ncanon counts the canonical products.
__global__ void k_row_thresholds(int64_t count, const int32_t *__restrict__ cu,
                                 const int32_t *__restrict__ cq, const int32_t *__restrict__ ci,
                                 const float *__restrict__ cx, const tc::RowBound *__restrict__ urb,
                                 const tc::RowBound *__restrict__ qrb, tc::Gacc gacc, float gcan,
                                 const float *__restrict__ U, const float *__restrict__ Q, int d,
                                 const int32_t *__restrict__ qself, float2 *__restrict__ thr,
                                 double *__restrict__ ths, int32_t *__restrict__ rself,
                                 unsigned long long *__restrict__ ncanon) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  bool canon = false;
  if (i < count) {
    const int64_t u = cu[i];
    const int q = cq[i];
    rself[i] = qself[q];
    const float x = cx ? cx[ci[i]] : __int_as_float(0x7fffffff);
    float2 t2 = make_float2(x, x);
    if (x == x) {
      const float b = tc::screen_bound_tc(urb[u], qrb[q], gacc, gcan);
      t2 = make_float2(__fsub_rd(x, b), __fadd_ru(x, b));
    }
    if (t2.x <= t2.y) {
      thr[i] = t2;
    } else {
      const double t = canon_dot(U + u * d, Q + (int64_t)q * d, d);
      thr[i] = make_float2(__double2float_rd(t), __double2float_ru(t));
      if (ths) ths[i] = t;
      canon = true;
    }
  }
  const int c = __popc(__ballot_sync(0xffffffffu, canon));
  if (c && (threadIdx.x & 31) == 0) atomicAdd(ncanon, (unsigned long long)c);
}

// Distinct users among the rows: a bit per user, counted when first set.
__global__ void k_distinct_users(int64_t count, const int32_t *__restrict__ cu,
                                 uint32_t *__restrict__ bits,
                                 unsigned long long *__restrict__ distinct) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  bool first = false;
  if (i < count) {
    const uint32_t u = (uint32_t)cu[i], b = 1u << (u & 31);
    first = !(bits[u >> 5] & b) && !(atomicOr(&bits[u >> 5], b) & b);
  }
  const int c = __popc(__ballot_sync(0xffffffffu, first));
  if (c && (threadIdx.x & 31) == 0) atomicAdd(distinct, (unsigned long long)c);
}

// Exact ranks of the candidates whose cu entry is valid (the others keep their
// ccount): compact them, canonical u.q, one tensor-core pass over P with a row per
// candidate (or, with rc_seg_min, per segment of a user's sorted thresholds).
// ccount[i] = #{p : s(u_i, p) > u_i.q_i}.
// With clb_all (bounds mode) items the screen cannot place are not resolved:
// ccount gets an upper and clb a lower bound of the count instead.  The
// single-product bounds pass takes a candidate's threshold from its screened score
// cx_all where it has one: the item bounds are some 50 times wider.
// With ncols > 0 only the first ncols items of the norm-sorted P are screened.
static rkr_status recount_candidates(const rkr_index *idx, const QueryCommon &qc, int64_t total,
                                     const int32_t *cu_all, const int32_t *cq_all,
                                     const float *cx_all,
                                     const int32_t *qself, uint32_t *ccount_all,
                                     uint32_t *clb_all, unsigned long long *ties_d,
                                     cudaStream_t st, int64_t *nusers = nullptr,
                                     int split = 1, int64_t ncols = 0,
                                     int64_t *ncanon = nullptr) {
  const float *Qd = qc.Qd;
  TcSide Pv = idx->Pt;   // a view: the same rows, possibly fewer of them
  if (ncols > 0 && ncols < Pv.rows) Pv.rows = ncols;
  const int bs = 256;
  DevBuf bcu, bcq, bci, bcc, bcur;
  int32_t *cu, *cq, *ci;
  uint32_t *ccount;
  unsigned long long *cur;
  RKR_TRY(tmp_alloc(bcur, &cur, 1, st));
  RKR_CUDA(cudaMemsetAsync(cur, 0, sizeof(unsigned long long), st));
  RKR_TRY(tmp_alloc(bcu, &cu, total, st));
  RKR_TRY(tmp_alloc(bcq, &cq, total, st));
  RKR_TRY(tmp_alloc(bci, &ci, total, st));
  {
    const int prof_slot = prof_begin("k_compact", st);
    k_compact<<<(unsigned)((total + bs - 1) / bs), bs, 0, st>>>(total, cu_all, cq_all, cur, cu, cq,
                                                                 ci);
    prof_end(prof_slot, st, 0.0);
  }
  note_launch();
  unsigned long long hc = 0;
  RKR_CUDA(cudaMemcpyAsync(&hc, cur, sizeof(hc), cudaMemcpyDeviceToHost, st));
  RKR_CUDA(cudaStreamSynchronize(st));
  const int64_t cnt = (int64_t)hc;
  if (cnt == 0) return RKR_OK;
  const char *span = ncols > 0   ? "span:recount(prefix)"
                     : clb_all ? (split ? "span:recount(bounds,split)" : "span:recount(bounds,single)")
                               : "span:recount(exact)";
  auto add_ties = [&](const int64_t *refined) -> rkr_status {
    if (!ties_d) return RKR_OK;
    // accumulate over chunks: [0] undecided items, [1] canonical evaluations
    unsigned long long t[2] = {0, 0};
    RKR_CUDA(cudaMemcpyAsync(t, ties_d, sizeof(t), cudaMemcpyDeviceToHost, st));
    RKR_CUDA(cudaStreamSynchronize(st));
    t[0] += (unsigned long long)refined[0];
    t[1] += (unsigned long long)refined[1];
    RKR_CUDA(cudaMemcpyAsync(ties_d, t, sizeof(t), cudaMemcpyHostToDevice, st));
    RKR_CUDA(cudaStreamSynchronize(st));
    return RKR_OK;
  };
  const unsigned blocks = (unsigned)((cnt + bs - 1) / bs);
  if (tuning().rc_seg_min == 0) {   // one row per candidate, in candidate order
    DevBuf b1, b2, b3, b4, b5, b6, b7;
    float2 *thr;
    double *ths = nullptr;
    int32_t *rself;
    uint32_t *lo, *hi = nullptr, *bits;
    unsigned long long *num;   // [0] canonical products, [1] distinct users
    RKR_TRY(tmp_alloc(b1, &thr, cnt, st));
    if (!clb_all) RKR_TRY(tmp_alloc(b2, &ths, cnt, st));
    RKR_TRY(tmp_alloc(b3, &rself, cnt, st));
    RKR_TRY(tmp_alloc(b4, &lo, cnt, st));
    if (clb_all) RKR_TRY(tmp_alloc(b5, &hi, cnt, st));
    RKR_TRY(tmp_alloc(b6, &num, 2, st));
    RKR_CUDA(cudaMemsetAsync(num, 0, 2 * sizeof(unsigned long long), st));
    RKR_CUDA(cudaMemsetAsync(lo, 0, sizeof(uint32_t) * cnt, st));
    if (hi) RKR_CUDA(cudaMemsetAsync(hi, 0, sizeof(uint32_t) * cnt, st));
    const float *cx = clb_all && !split ? cx_all : nullptr;
    {
      const int prof_slot = prof_begin("k_row_thresholds", st);
      k_row_thresholds<<<blocks, bs, 0, st>>>(cnt, cu, cq, ci, cx, idx->Ut.rb3, qc.Qt.rb3,
                                              tc_gacc(idx->Ut.kp, 1), tc_gcan(idx->d), idx->U, Qd,
                                              idx->d, qself, thr, ths, rself, num);
      prof_end(prof_slot, st, 0.0);
    }
    note_launch();
    RKR_CUDA(cudaGetLastError());
    if (nusers) {
      const size_t words = (size_t)(idx->n + 31) / 32;
      RKR_TRY(tmp_alloc(b7, &bits, words, st));
      RKR_CUDA(cudaMemsetAsync(bits, 0, sizeof(uint32_t) * words, st));
      k_distinct_users<<<blocks, bs, 0, st>>>(cnt, cu, bits, num + 1);
      note_launch();
      RKR_CUDA(cudaGetLastError());
    }
    int64_t refined[2] = {0, 0};
    {
      ProfScope prof(span, st, 0.0);
      RKR_TRY(tc_recount(idx, idx->Ut, Pv, cnt, cnt, nullptr, nullptr, cu, rself, thr, ths, lo, hi,
                         st, refined, split));
    }
    RKR_TRY(add_ties(refined));
    unsigned long long hn[2] = {0, 0};
    RKR_CUDA(cudaMemcpyAsync(hn, num, sizeof(hn), cudaMemcpyDeviceToHost, st));
    k_scatter_back<<<blocks, bs, 0, st>>>(cnt, ci, clb_all ? hi : lo, ccount_all);
    note_launch();
    if (clb_all) {
      k_scatter_back<<<blocks, bs, 0, st>>>(cnt, ci, lo, clb_all);
      note_launch();
    }
    RKR_CUDA(cudaGetLastError());
    RKR_CUDA(cudaStreamSynchronize(st));
    if (ncanon) *ncanon += (int64_t)hn[0];
    if (nusers) *nusers += (int64_t)hn[1];
    return RKR_OK;
  }
  if (ncanon) *ncanon += cnt;   // k_cand_theta forms each row's canonical u.q
  RKR_TRY(tmp_alloc(bcc, &ccount, cnt, st));
  int64_t Np2 = 1;
  while (Np2 < cnt) Np2 <<= 1;
  DevBuf b1, b2, b3, b4, b5, b6, b7, b8, b9;
  double *th, *ths;
  uint64_t *khi, *klo;
  int32_t *val, *slen;
  int64_t *sstart;
  uint32_t *hist;
  unsigned long long *nseg_d;
  RKR_TRY(tmp_alloc(b1, &th, cnt, st));
  RKR_TRY(tmp_alloc(b2, &khi, Np2, st));
  RKR_TRY(tmp_alloc(b3, &klo, Np2, st));
  RKR_TRY(tmp_alloc(b4, &val, Np2, st));
  RKR_TRY(tmp_alloc(b5, &sstart, cnt, st));
  RKR_TRY(tmp_alloc(b6, &slen, cnt, st));
  RKR_TRY(tmp_alloc(b7, &hist, 2 * cnt, st));
  RKR_TRY(tmp_alloc(b8, &ths, cnt, st));
  RKR_TRY(tmp_alloc(b9, &nseg_d, 3, st));
  {
    const int prof_slot = prof_begin("k_cand_theta", st);
    k_cand_theta<<<(unsigned)((Np2 + bs - 1) / bs), bs, 0, st>>>(cnt, cu, cq, idx->U, Qd, idx->d,
                                                                  th, khi, klo, val, Np2);
    prof_end(prof_slot, st, 0.0);
  }
  note_launch();
  RKR_CUDA(cudaGetLastError());
  RKR_TRY(bitonic_sort(Sort128{khi, klo, val}, Np2, "k_sort<128>", st));
  RKR_CUDA(cudaMemsetAsync(nseg_d, 0, 3 * sizeof(unsigned long long), st));
  RKR_CUDA(cudaMemsetAsync(slen, 0, sizeof(int32_t) * cnt, st));
  k_segments<<<(unsigned)((cnt + bs - 1) / bs), bs, 0, st>>>(cnt, khi, tuning().rc_seg_min,
                                                              nseg_d, sstart, slen);
  note_launch();
  RKR_CUDA(cudaGetLastError());
  unsigned long long segu[3] = {0, 0, 0};
  RKR_CUDA(cudaMemcpyAsync(segu, nseg_d, sizeof(segu), cudaMemcpyDeviceToHost, st));
  RKR_CUDA(cudaStreamSynchronize(st));
  const int64_t n1 = (int64_t)segu[0], n2 = (int64_t)segu[2], off2 = cnt - n2;
  if (nusers) *nusers += (int64_t)segu[1];
  // per segment slot (front range: one threshold; back range: several)
  DevBuf b10, b11, b12, b13, b14;
  int32_t *suser, *sself, *scol, *spos;
  float2 *thr;
  RKR_TRY(tmp_alloc(b14, &thr, cnt, st));
  RKR_TRY(tmp_alloc(b10, &suser, cnt, st));
  RKR_TRY(tmp_alloc(b11, &sself, cnt, st));
  RKR_TRY(tmp_alloc(b12, &scol, cnt, st));
  RKR_TRY(tmp_alloc(b13, &spos, cnt, st));
  k_seg_prep<<<(unsigned)((cnt + bs - 1) / bs), bs, 0, st>>>(
      cnt, sstart, slen, khi, val, th, cq, qself, suser, sself, thr, ths, hist, scol, spos);
  note_launch();
  RKR_CUDA(cudaGetLastError());
  int64_t refined[2] = {0, 0};
  DevBuf bhh;
  uint32_t *hist_hi = nullptr;
  if (clb_all) {
    RKR_TRY(tmp_alloc(bhh, &hist_hi, 2 * cnt, st));
    RKR_CUDA(cudaMemsetAsync(hist_hi, 0, sizeof(uint32_t) * 2 * cnt, st));
  }
  {
    ProfScope prof(span, st, 0.0);
    if (n1 > 0)
      RKR_TRY(tc_recount(idx, idx->Ut, Pv, n1, cnt, sstart, slen, suser, sself, thr, ths, hist,
                         hist_hi, st, refined, split));
    if (n2 > 0) {
      int64_t ref2[2] = {0, 0};
      RKR_TRY(tc_recount(idx, idx->Ut, Pv, n2, cnt, sstart + off2, slen + off2,
                         suser + off2, sself + off2, thr, ths, hist, hist_hi, st, ref2, split,
                         scol, spos));
      refined[0] += ref2[0];
      refined[1] += ref2[1];
    }
  }
  const int64_t nseg = cnt;   // the kernels below walk every slot and skip the empty ones
  {
    const int prof_slot = prof_begin("k_seg_suffix", st);
    k_seg_suffix<<<(unsigned)((nseg + bs - 1) / bs), bs, 0, st>>>((int64_t)nseg, sstart, slen,
                                                                   hist);
    prof_end(prof_slot, st, 0.0);
  }
  note_launch();
  RKR_CUDA(cudaGetLastError());
  RKR_TRY(add_ties(refined));
  {
    const int prof_slot = prof_begin("k_scatter_counts", st);
    k_scatter_counts<<<(unsigned)((nseg + bs - 1) / bs), bs, 0, st>>>((int64_t)nseg, sstart, slen,
                                                                     val, hist, ccount);
    prof_end(prof_slot, st, 0.0);
  }
  note_launch();
  if (clb_all) {  // lower ends into clb, upper ends (below) into ccount
    k_scatter_back<<<(unsigned)((cnt + bs - 1) / bs), bs, 0, st>>>(cnt, ci, ccount, clb_all);
    note_launch();
    k_seg_suffix<<<(unsigned)((nseg + bs - 1) / bs), bs, 0, st>>>((int64_t)nseg, sstart, slen,
                                                                   hist_hi);
    note_launch();
    k_scatter_counts<<<(unsigned)((nseg + bs - 1) / bs), bs, 0, st>>>((int64_t)nseg, sstart,
                                                                     slen, val, hist_hi, ccount);
    note_launch();
  }
  k_scatter_back<<<(unsigned)((cnt + bs - 1) / bs), bs, 0, st>>>(cnt, ci, ccount, ccount_all);
  note_launch();
  RKR_CUDA(cudaGetLastError());
  return RKR_OK;
}

// Candidates whose count interval has closed (lower == upper) need no recount.
__global__ void k_drop_decided(int64_t n, const uint32_t *__restrict__ ccount,
                               const uint32_t *__restrict__ clb, int32_t *__restrict__ cu_fb) {
  int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i < n && cu_fb[i] >= 0 && ccount[i] == clb[i]) cu_fb[i] = -1;
}

static rkr_status count_valid(const int32_t *v, int64_t n, unsigned long long *out,
                              cudaStream_t st) {
  DevBuf b;
  unsigned long long *d;
  RKR_TRY(tmp_alloc(b, &d, 1, st));
  RKR_CUDA(cudaMemsetAsync(d, 0, sizeof(unsigned long long), st));
  k_count_valid<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(n, v, d);
  note_launch();
  RKR_CUDA(cudaMemcpyAsync(out, d, sizeof(unsigned long long), cudaMemcpyDeviceToHost, st));
  RKR_CUDA(cudaStreamSynchronize(st));
  return RKR_OK;
}

// Interval [lo, hi] of a candidate's u.q in float: from its screened score, or from
// the compensated product of its rows.  False when an end is not finite (products of
// the rows beyond the range of float): such a candidate takes no part in the grid.
__device__ __forceinline__ bool cand_interval(int64_t u, int q, float x,
                                              const tc::RowBound *__restrict__ urb,
                                              const tc::RowBound *__restrict__ qrb, tc::Gacc gacc,
                                              float gcan, const float *__restrict__ U,
                                              const float *__restrict__ Q, int d, float &lo,
                                              float &hi) {
  if (x == x) {
    const float b = tc::screen_bound_tc(urb[u], qrb[q], gacc, gcan);
    lo = __fsub_rd(x, b);
    hi = __fadd_ru(x, b);
  } else {
    dot2_interval_f(U + u * d, Q + (int64_t)q * d, d, lo, hi);
  }
  return lo > -INFINITY && hi < INFINITY;   // (a NaN end fails both)
}

// Order-preserving 32-bit key of a float, and its inverse.
__device__ __forceinline__ uint32_t float_key(float x) {
  const uint32_t b = __float_as_uint(x);
  return (b >> 31) ? ~b : (b | 0x80000000u);
}
__device__ __forceinline__ float key_float(uint32_t k) {
  return __uint_as_float((k >> 31) ? (k & 0x7fffffffu) : ~k);
}

// Range of the open candidates' u.q per user, as keys (kmin starts at ~0, the key of
// no finite value, kmax at 0).
__global__ void k_open_range(int64_t cnt, const int32_t *__restrict__ cu_fb,
                             const int32_t *__restrict__ cq, const float *__restrict__ cx,
                             const tc::RowBound *__restrict__ urb,
                             const tc::RowBound *__restrict__ qrb, tc::Gacc gacc, float gcan,
                             const float *__restrict__ U, const float *__restrict__ Q, int d,
                             uint32_t *__restrict__ kmin, uint32_t *__restrict__ kmax) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= cnt) return;
  const int64_t u = cu_fb[i];
  if (u < 0) return;
  float lo, hi;
  if (!cand_interval(u, cq[i], cx[i], urb, qrb, gacc, gcan, U, Q, d, lo, hi)) return;
  const uint32_t a = float_key(lo), b = float_key(hi);
  if (a < kmin[u]) atomicMin(&kmin[u], a);
  if (b > kmax[u]) atomicMax(&kmax[u], b);
}

// Users with open candidates, each with a grid from its smallest to its largest u.q.
__global__ void k_grid_users(int64_t n, const uint32_t *__restrict__ kmin,
                             const uint32_t *__restrict__ kmax, const float *__restrict__ unrm,
                             unsigned long long *__restrict__ cursor, int32_t *__restrict__ ulist,
                             int32_t *__restrict__ uslot, double *__restrict__ yg0,
                             double *__restrict__ ymax, float *__restrict__ ytop,
                             float *__restrict__ ybot, float *__restrict__ nrm) {
  const int64_t u = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const bool has = u < n && kmin[u] != 0xffffffffu;
  const unsigned act = __ballot_sync(0xffffffffu, has);
  if (!has) return;
  const int lane = threadIdx.x & 31, leader = __ffs(act) - 1;
  unsigned long long base = 0;
  if (lane == leader) base = atomicAdd(cursor, (unsigned long long)__popc(act));
  base = __shfl_sync(act, base, leader);
  const int64_t s = (int64_t)base + __popc(act & ((1u << lane) - 1u));
  const float lo = key_float(kmin[u]), hi = key_float(kmax[u]);
  ulist[s] = (int32_t)u;
  uslot[u] = (int32_t)s;
  yg0[s] = (double)lo;
  ymax[s] = (double)hi;
  ytop[s] = hi;
  ybot[s] = lo;
  nrm[s] = unrm[u];
}

// Count bounds of the open candidates from their user's grid: u.q >= y_{jl - 1} and
// u.q < y_{jh} give CLO[jh] <= count <= CHI[jl - 1].
__global__ void k_grid_bound(int64_t cnt, const int32_t *__restrict__ cu_fb,
                             const int32_t *__restrict__ cq, const float *__restrict__ cx,
                             const tc::RowBound *__restrict__ urb,
                             const tc::RowBound *__restrict__ qrb, tc::Gacc gacc, float gcan,
                             const float *__restrict__ U, const float *__restrict__ Q, int d,
                             const int32_t *__restrict__ uslot, const BinFP *__restrict__ ybin,
                             const uint32_t *__restrict__ CLO,
                             const uint32_t *__restrict__ CHI, uint32_t *__restrict__ ccount,
                             uint32_t *__restrict__ clb) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= cnt) return;
  const int64_t u = cu_fb[i];
  if (u < 0) return;
  float lo, hi;
  if (!cand_interval(u, cq[i], cx[i], urb, qrb, gacc, gcan, U, Q, d, lo, hi)) return;
  const int64_t s = uslot[u];   // set: k_open_range saw this finite interval
  const TightBins tb(ybin[s]);
  if (!tb.usable()) return;   // a grid without a usable step bounds nothing
  const int jl = tb.lo(lo, kDGrid), jh = tb.hi(hi, kDGrid);
  if (jl >= 1) ccount[i] = min(ccount[i], CHI[s * kDGrid + jl - 1]);
  if (jh < kDGrid) clb[i] = max(clb[i], CLO[s * kDGrid + jh]);
}

// When a chunk's open candidates (h of them) are many per user, their counts are
// first bounded together: one single-product screen of the users concerned against
// P counts each user's scores on a grid of kDGrid points spanning its candidates'
// u.q, and the cap (k-th smallest count upper bound) then drops most of them.  A
// grid row costs about six recount rows (every score inside the grid goes to two
// histograms), so it is built from kGridPerUser candidates per user on, where it
// can save a recount of each.  *h is the number still open on return.  Nothing
// happens when the scratch cannot be had.
constexpr int64_t kGridPerUser = 12;
constexpr int64_t kGridMinRows = (int64_t)1 << 16;

static rkr_status grid_prune(const rkr_index *idx, const QueryCommon &qc, int qa, int qb,
                             int64_t cnt, const int64_t *qoff_rel, const uint32_t *cursor,
                             const int32_t *cq, const float *cx, uint32_t *ccount, uint32_t *clb,
                             int32_t *cu_fb, unsigned long long *h, cudaStream_t st) {
  const int64_t n = idx->n;
  const tc::Gacc gacc = tc_gacc(idx->Ut.kp, 1);
  const float gcan = tc_gcan(idx->d);
  DevBuf b[13];
  bool ok = true;
  auto get = [&](int i, auto **p, size_t count) {
    if (!ok) return;
    if (pool_malloc_async((void **)p, count * sizeof(**p), st) != cudaSuccess) {
      cudaGetLastError();
      ok = false;
      return;
    }
    b[i].p = (void *)*p;
    b[i].st = st;
  };
  uint32_t *kmin = nullptr, *kmax = nullptr;
  int32_t *ulist = nullptr, *uslot = nullptr;
  double *yg0 = nullptr, *ymax = nullptr, *ydx = nullptr;
  float *ytop = nullptr, *ybot = nullptr, *nrm = nullptr;
  unsigned long long *num = nullptr;
  get(0, &kmin, n);
  get(1, &kmax, n);
  get(2, &num, 1);
  if (!ok) return RKR_OK;
  RKR_CUDA(cudaMemsetAsync(kmin, 0xff, sizeof(uint32_t) * n, st));
  RKR_CUDA(cudaMemsetAsync(kmax, 0, sizeof(uint32_t) * n, st));
  RKR_CUDA(cudaMemsetAsync(num, 0, sizeof(unsigned long long), st));
  const unsigned cblocks = (unsigned)((cnt + 255) / 256), ublocks = (unsigned)((n + 255) / 256);
  k_open_range<<<cblocks, 256, 0, st>>>(cnt, cu_fb, cq, cx, idx->Ut.rb3, qc.Qt.rb3, gacc, gcan,
                                        idx->U, qc.Qd, idx->d, kmin, kmax);
  note_launch();
  get(3, &ulist, n);
  get(4, &uslot, n);
  get(5, &yg0, n);
  get(6, &ymax, n);
  get(7, &ytop, n);
  get(8, &ybot, n);
  get(9, &nrm, n);
  if (!ok) return RKR_OK;
  k_grid_users<<<ublocks, 256, 0, st>>>(n, kmin, kmax, idx->unrm, num, ulist, uslot, yg0, ymax,
                                        ytop, ybot, nrm);
  note_launch();
  RKR_CUDA(cudaGetLastError());
  unsigned long long users = 0;
  RKR_CUDA(cudaMemcpyAsync(&users, num, sizeof(users), cudaMemcpyDeviceToHost, st));
  RKR_CUDA(cudaStreamSynchronize(st));
  if (users == 0 || *h < (unsigned long long)kGridPerUser * users) return RKR_OK;
  const int64_t nu = (int64_t)users;
  BinFP *ybin = nullptr;
  uint32_t *CLO = nullptr, *CHI = nullptr;
  DevBuf bb;
  get(10, &ydx, nu);
  get(11, &CLO, nu * kDGrid);
  get(12, &CHI, nu * kDGrid);
  if (ok && pool_malloc_async(&ybin, sizeof(BinFP) * nu, st) == cudaSuccess) {
    bb.p = ybin;
    bb.st = st;
  } else {
    cudaGetLastError();
    return RKR_OK;
  }
  RKR_TRY(make_binfp_rows(nu, nrm, yg0, ymax, kDGrid, idx->pmax, ydx, ybin, st));
  TcSide A;
  if (tc_gather_side(idx->Ut, ulist, nu, false, A, st) != RKR_OK) {
    set_error("%s", "");
    return RKR_OK;
  }
  const rkr_status gs =
      tc_count_grid(idx, A, idx->Pt, CountGrid{ybin, yg0, ytop, ybot, CLO, CHI}, st);
  tc_gather_free(A, st);
  RKR_TRY(gs);
  k_grid_bound<<<cblocks, 256, 0, st>>>(cnt, cu_fb, cq, cx, idx->Ut.rb3, qc.Qt.rb3, gacc, gcan,
                                        idx->U, qc.Qd, idx->d, uslot, ybin, CLO, CHI, ccount,
                                        clb);
  note_launch();
  {
    const int prof_slot = prof_begin("k_recount_filter", st);
    k_recount_filter<<<qb - qa, filter_threads(cnt, qb - qa), 0, st>>>(qa, qoff_rel, cursor, qc.kq_d, ccount,
                                                         clb, cu_fb, (uint32_t)idx->m);
    prof_end(prof_slot, st, 0.0);
  }
  note_launch();
  k_drop_decided<<<cblocks, 256, 0, st>>>(cnt, ccount, clb, cu_fb);
  note_launch();
  RKR_CUDA(cudaGetLastError());
  return count_valid(cu_fb, cnt, h, st);
}

// Early termination over the norm-sorted items (tuning rc_prefix; Alg. 1 sorts P
// by descending norm).  For the queries with many candidates still to recount,
// every such candidate is first screened against the first m1 items only: its
// certain count there is a lower bound of its count over P, and its possible
// count there ranks how promising it is.  The query's most promising candidates
// are recounted over all of P, the cap (k-th smallest count upper bound) is taken
// again, and every other candidate whose prefix lower bound exceeds the cap is
// dropped unrecounted: it cannot be among the k smallest ranks.  The rest go back
// to the recount.  On return *h2 is the number of candidates still to recount.
static rkr_status prefix_prune(const rkr_index *idx, const QueryCommon &qc, int qa, int qb,
                               int64_t cnt, const int64_t *qoff_rel, const uint32_t *cursor,
                               const int32_t *cq, const float *cx, const int32_t *qself,
                               uint32_t *ccount, uint32_t *clb, int32_t *cu_fb,
                               int64_t *recount_users,
                               unsigned long long *h2, int64_t *rows, int64_t *pruned,
                               int64_t *ncanon, cudaStream_t st) {
  const int64_t m1 = idx->m / tuning().rc_prefix / 256 * 256;
  if (m1 < 256 || m1 >= idx->m) return RKR_OK;
  DevBuf b1, b2, b3, b4, b5;
  int32_t *cu_pre, *cu_park;
  uint32_t *hi1, *lo1;
  unsigned long long *npre_d, npre = 0;
  RKR_TRY(tmp_alloc(b1, &cu_pre, cnt, st));
  RKR_TRY(tmp_alloc(b2, &cu_park, cnt, st));
  RKR_TRY(tmp_alloc(b3, &hi1, cnt, st));
  RKR_TRY(tmp_alloc(b4, &lo1, cnt, st));
  RKR_TRY(tmp_alloc(b5, &npre_d, 1, st));
  RKR_CUDA(cudaMemsetAsync(cu_pre, 0xff, sizeof(int32_t) * cnt, st));
  RKR_CUDA(cudaMemsetAsync(cu_park, 0xff, sizeof(int32_t) * cnt, st));
  RKR_CUDA(cudaMemsetAsync(hi1, 0xff, sizeof(uint32_t) * cnt, st));
  RKR_CUDA(cudaMemsetAsync(lo1, 0, sizeof(uint32_t) * cnt, st));
  RKR_CUDA(cudaMemsetAsync(npre_d, 0, sizeof(unsigned long long), st));
  k_prefix_split<<<qb - qa, 256, 0, st>>>(qa, qoff_rel, cursor, qc.kq_d, cu_fb, cu_pre, npre_d);
  note_launch();
  RKR_CUDA(cudaGetLastError());
  RKR_CUDA(cudaMemcpyAsync(&npre, npre_d, sizeof(npre), cudaMemcpyDeviceToHost, st));
  RKR_CUDA(cudaStreamSynchronize(st));
  if (npre == 0) return RKR_OK;
  *rows += (int64_t)npre;
  // certain (lo1) and possible (hi1) counts over the prefix, single product
  RKR_TRY(recount_candidates(idx, qc, cnt, cu_pre, cq, cx, qself, hi1, lo1, nullptr, st, nullptr,
                             0, m1, ncanon));
  k_prefix_pick<<<qb - qa, filter_threads(cnt, qb - qa), 0, st>>>(qa, qoff_rel, cursor, qc.kq_d, cu_pre, hi1, lo1, clb,
                                          cu_fb, cu_park);
  note_launch();
  RKR_CUDA(cudaGetLastError());
  unsigned long long parked = 0, kept = 0, h = 0;
  RKR_TRY(count_valid(cu_park, cnt, &parked, st));
  RKR_TRY(count_valid(cu_fb, cnt, &h, st));
  if (h > 0)  // the promising rows and the other queries' rows, over all of P
    RKR_TRY(recount_candidates(idx, qc, cnt, cu_fb, cq, cx, qself, ccount, clb, nullptr, st,
                               recount_users, tuning().rc_single_first ? 0 : 1, 0, ncanon));
  {
    const int prof_slot = prof_begin("k_recount_filter", st);
    k_recount_filter<<<qb - qa, filter_threads(cnt, qb - qa), 0, st>>>(qa, qoff_rel, cursor, qc.kq_d, ccount, clb, cu_fb,
                                                         (uint32_t)idx->m);
    k_recount_filter<<<qb - qa, filter_threads(cnt, qb - qa), 0, st>>>(qa, qoff_rel, cursor, qc.kq_d, ccount, clb,
                                                         cu_park, (uint32_t)idx->m);
    prof_end(prof_slot, st, 0.0);
  }
  note_launch();
  note_launch();
  k_drop_decided<<<(unsigned)((cnt + 255) / 256), 256, 0, st>>>(cnt, ccount, clb, cu_fb);
  note_launch();
  RKR_CUDA(cudaGetLastError());
  RKR_TRY(count_valid(cu_park, cnt, &kept, st));
  *pruned += (int64_t)(parked - kept);
  k_prefix_unpark<<<(unsigned)((cnt + 255) / 256), 256, 0, st>>>(cnt, cu_park, cu_fb);
  note_launch();
  RKR_CUDA(cudaGetLastError());
  RKR_TRY(count_valid(cu_fb, cnt, h2, st));
  return RKR_OK;
}

// Steps 2-3 of queries qa .. qa + nblocks - 1 (one CTA each).
static rkr_status select_approx(int qa, int nblocks, const int64_t *qoff, const uint32_t *qcount,
                                const ApproxCand &C, const int32_t *kq, double c,
                                const int64_t *out_off, int32_t *users_d, uint32_t *nlo_d,
                                uint32_t *nup_d, double *est_d, int32_t *case_d, int32_t *nc_d,
                                int *err, cudaStream_t st, const rkr_index *idx) {
  const bool few = nblocks <= sm_count();
  auto kern = few ? k_select_approx<kSelThreadsFew> : k_select_approx<kSelThreads>;
  const size_t sm = select_smem(few, idx->d);
  RKR_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)select_smem(few, kMaxD)));
  const int prof_slot = prof_begin("k_select_approx", st);
  kern<<<nblocks, few ? kSelThreadsFew : kSelThreads, sm, st>>>(
      qa, qoff, qcount, C, kq, c, (uint32_t)idx->s, idx->tau, idx->fmin, idx->delta, out_off,
      users_d, nlo_d, nup_d, est_d, case_d, nc_d, err, (uint32_t)(idx->m * idx->s),
      user_bits(idx->n));
  prof_end(prof_slot, st, 0.0);
  note_launch();
  RKR_CUDA(cudaGetLastError());
  return RKR_OK;
}

rkr_status run_query_approx(const rkr_index *idx, const QueryCommon &qc, int nq, double c,
                            int32_t *users_d, uint32_t *nlo_d, uint32_t *nup_d, double *est_d,
                            int32_t *case_d, int32_t *nc_d, rkr_query_stats *stats,
                            cudaStream_t st) {
  DevBuf bn, bcap;
  int32_t *lstar_d;
  int64_t *ncand_d;
  uint32_t *cap_d;
  RKR_TRY(tmp_alloc(bn, (char **)&ncand_d, plan_bytes(nq), st));
  lstar_d = (int32_t *)(ncand_d + nq);
  RKR_TRY(tmp_alloc(bcap, &cap_d, nq, st));
  DevBuf bw;
  CallWords *words;
  RKR_TRY(words_alloc(bw, &words, st));
  unsigned long long *nfp64_d = &words->nfp64;
  Plan plan;
  double ms_theta = 0.0, ms_res = 0.0, ms_sel = 0.0;
  SpanClock clk(st);
  const int t1 = clk.begin(&ms_theta);
  const Grid grid{qc.bf,  idx->fmin, idx->tau, idx->JU, idx->JL, idx->nlev_a,
                  idx->N, idx->N,    (uint32_t)(idx->m * idx->s), (uint32_t)idx->s};
  RKR_TRY(screen_plan(idx, qc, nq, grid, st, lstar_d, cap_d, ncand_d, plan));
  clk.end(t1);
  int wide = 0;
  for (int q = 0; q < nq; ++q) wide += plan.lstar[q] >= idx->nlev_a - 1;
  std::vector<int64_t> qoff(nq + 1, 0);
  for (int q = 0; q < nq; ++q) qoff[q + 1] = qoff[q] + plan.ncand[q];
  DevBuf bo;
  int64_t *qoff_d;
  RKR_TRY(tmp_alloc(bo, &qoff_d, nq + 1, st));
  std::vector<std::vector<int64_t>> rels;   // per chunk, copied from until the call settles
  StreamGuard guard(st);
  RKR_CUDA(cudaMemcpyAsync(qoff_d, qoff.data(), sizeof(int64_t) * (nq + 1),
                           cudaMemcpyHostToDevice, st));
  for (auto ch : chunk_queries(plan.ncand, candidate_budget())) {
    int qa = ch.first, qb = ch.second;
    int64_t cnt = qoff[qb] - qoff[qa];
    DevBuf b1, b2, b3, b4, b5, b6, b7, b8, b9;
    int32_t *cu, *cq, *cj;
    uint32_t *cursor, *nlo, *nup;
    double *th;
    float *cx;
    int64_t *qoff_rel;
    RKR_TRY(tmp_alloc(b9, &cx, cnt, st));
    RKR_CUDA(cudaMemsetAsync(cx, 0xff, sizeof(float) * std::max<int64_t>(cnt, 1), st));  // NaN
    RKR_TRY(tmp_alloc(b1, &cu, cnt, st));
    RKR_TRY(tmp_alloc(b2, &cq, cnt, st));
    RKR_TRY(tmp_alloc(b3, &cursor, nq, st));
    RKR_TRY(tmp_alloc(b4, &th, cnt, st));
    RKR_TRY(tmp_alloc(b5, &cj, cnt, st));
    RKR_TRY(tmp_alloc(b6, &nlo, cnt, st));
    RKR_TRY(tmp_alloc(b7, &nup, cnt, st));
    RKR_TRY(tmp_alloc(b8, &qoff_rel, nq + 1, st));
    // offsets relative to the chunk start, so candidate arrays hold only this chunk
    rels.emplace_back(nq + 1, 0);
    std::vector<int64_t> &rel = rels.back();
    for (int q = 0; q <= nq; ++q) rel[q] = qoff[q] - qoff[qa];
    RKR_CUDA(cudaMemcpyAsync(qoff_rel, rel.data(), sizeof(int64_t) * (nq + 1),
                             cudaMemcpyHostToDevice, st));
    RKR_CUDA(cudaMemsetAsync(cursor, 0, sizeof(uint32_t) * nq, st));
    RKR_CUDA(cudaMemsetAsync(cu, 0xff, sizeof(int32_t) * std::max<int64_t>(cnt, 1), st));
    const int t2 = clk.begin(&ms_theta);
    RKR_TRY(emit_candidates(idx, qc, qa, qb, grid, plan, lstar_d, cap_d, qoff_rel, cursor, cu, cq,
                            cx, true, words, st));
    clk.end(t2);
    const int t3 = clk.begin(&ms_res);
    if (cnt > 0) {
      {
        const int prof_slot = prof_begin("k_resolve_approx", st);
        k_resolve_approx<<<(unsigned)((cnt + 127) / 128), 128, 0, st>>>(
            cnt, cu, cq, cx, idx->Ut.rb3, qc.Qt.rb3, tc_gacc(idx->Ut.kp, 1), tc_gcan(idx->d),
            idx->U, qc.Qd, idx->d, idx->fmin, idx->delta, qc.bf, idx->N, idx->tau,
            (uint32_t)(idx->m * idx->s), th, cj, nlo, nup, nfp64_d);
        prof_end(prof_slot, st, 0.0);
        note_launch();
      }
      RKR_CUDA(cudaGetLastError());
    }
    clk.end(t3);
    const int t4 = clk.begin(&ms_sel);
    RKR_TRY(select_approx(qa, qb - qa, qoff_rel, cursor,
                          ApproxCand{cu, nlo, nup, th, cj, idx->U, qc.Qd, idx->d, nfp64_d},
                          qc.kq_d, c, qc.out_off_d, users_d, nlo_d, nup_d, est_d, case_d, nc_d,
                          &words->select_err, st, idx));
    clk.end(t4);
  }
  CallWords hw;
  RKR_TRY(words_check(words, hw, st));
  guard.settled = true;
  clk.finish();
  if (stats) {
    stats->pairs = idx->n * (int64_t)nq;
    stats->candidates = (int64_t)hw.candidates;
    stats->fp64_dots = (int64_t)hw.nfp64;
    stats->near_ties = 0;
    stats->wide_queries = wide;
    stats->deep_queries = (int32_t)plan.deep.size();
    stats->ms_theta = ms_theta;
    stats->ms_resolve = ms_res;
    stats->ms_select = ms_sel;
  }
  return RKR_OK;
}

rkr_status launch_select_approx(int qa, int nblocks, const int64_t *qoff, const uint32_t *qcount,
                                const int32_t *uid, const uint32_t *nlo, const uint32_t *nup,
                                double *th, const int32_t *cj, const float *Qd,
                                const int32_t *kq, double c, const int64_t *out_off,
                                int32_t *users_d, uint32_t *nlo_d, uint32_t *nup_d, double *est_d,
                                int32_t *case_d, int32_t *nc_d, int *err, cudaStream_t st,
                                const rkr_index *idx) {
  return select_approx(qa, nblocks, qoff, qcount,
                       ApproxCand{uid, nlo, nup, th, cj, idx->U, Qd, idx->d, nullptr}, kq, c,
                       out_off, users_d, nlo_d, nup_d, est_d, case_d, nc_d, err, st, idx);
}

struct LearnedPrune {
  rkr_pruner *pr;
  const float *Xu;   // per-user features
  const int32_t *keep;  // candidates kept per query (device, nq)
  int certify;          // 1: exact fallback for cut candidates that could still matter
  bool table;           // predictions from the pruner's per-user tables
};

constexpr int64_t kLearnedUncut = 32;

// Per query (one block), among the candidates still to be recounted (fb >= 0):
// those whose predicted log rank y is above the keep[q]-th smallest prediction
// are cut (fb = cu = -1, count = the largest key, so selection never takes them).
// Candidates whose exact count is known already are not touched.
__global__ void __launch_bounds__(kFilterThreads)
    k_learned_cut(int qa, const int64_t *__restrict__ qoff, const uint32_t *__restrict__ qcount,
                  const int32_t *__restrict__ keep_q, const float *__restrict__ y,
                  int32_t *__restrict__ fb_all, int32_t *__restrict__ cu_all,
                  uint32_t *__restrict__ ccount, int32_t *__restrict__ cutu_all,
                  int64_t n_users, unsigned long long *__restrict__ ncut) {
  __shared__ __align__(16) uint32_t hist[256];
  __shared__ uint64_t bc[2];
  __shared__ unsigned long long acc;
  const int q = qa + blockIdx.x;
  const int64_t base = qoff[q] - qoff[qa];
  const int64_t cnt = qcount[q];
  const int64_t keep = keep_q[q];
  int32_t *fb = fb_all + base, *cu = cu_all + base, *cutu = cutu_all + base;
  uint32_t *cc = ccount + base;
  const float *yy = y + base;
  auto key_of = [&](int64_t i) {
    const uint32_t b = __float_as_uint(yy[i]);
    return (uint64_t)((b & 0x80000000u) ? ~b : (b | 0x80000000u));
  };
  const int64_t open = block_count(cnt, [&](int64_t i) { return fb[i] >= 0; }, &acc);
  // a query whose candidates to recount are a large part of all users and far more
  // than it keeps is left uncut: such candidates have weak rank lower bounds (u.q
  // lies below the tail lists) and the exact fallback would revive them anyway
  if (open <= keep || (n_users > 0 && open > kLearnedUncut * keep && open > n_users / 4)) return;
  const uint64_t kth = block_kth(cnt, (uint64_t)keep, 32,
                                 [&](int64_t i, uint64_t &key) {
                                   if (fb[i] < 0) return false;
                                   key = key_of(i);
                                   return true;
                                 },
                                 hist, bc);
  __syncthreads();
  const int64_t cut = block_count(cnt, [&](int64_t i) { return fb[i] >= 0 && key_of(i) > kth; },
                                  &acc);
  for (int64_t i = threadIdx.x; i < cnt; i += blockDim.x)
    if (fb[i] >= 0 && key_of(i) > kth) {
      cutu[i] = cu[i];   // kept for the exact fallback
      fb[i] = -1;
      cu[i] = -1;
      cc[i] = 0xffffffffu;
    }
  if (threadIdx.x == 0) atomicAdd(ncut, (unsigned long long)cut);
}

// Exact fallback of the learned cut (one block per query).  cap = the k-th
// smallest count among the candidates not cut, an upper bound of the k-th
// smallest count of all candidates.  A cut candidate whose lower bound clb is at
// most cap could still be among the k best: it is revived (its user restored and
// sent to the recount).  The others have count >= clb > cap and cannot be.
__global__ void __launch_bounds__(256)
    k_learned_revive(int qa, const int64_t *__restrict__ qoff,
                     const uint32_t *__restrict__ qcount, const int32_t *__restrict__ kq,
                     const uint32_t *__restrict__ ccount, const uint32_t *__restrict__ clb,
                     int32_t *__restrict__ fb_all, int32_t *__restrict__ cu_all,
                     int32_t *__restrict__ cutu_all, unsigned long long *__restrict__ nrev) {
  __shared__ __align__(16) uint32_t hist[256];
  __shared__ uint64_t bc[2];
  __shared__ unsigned long long acc;
  const int q = qa + blockIdx.x;
  const int64_t base = qoff[q] - qoff[qa];
  const int64_t cnt = qcount[q];
  const int k = kq[q];
  if (cnt < k) return;
  int32_t *fb = fb_all + base, *cu = cu_all + base, *cutu = cutu_all + base;
  const uint32_t *cc = ccount + base, *lb = clb + base;
  const uint64_t cap = block_kth(cnt, (uint64_t)k, 32,
                                 [&](int64_t i, uint64_t &key) { key = cc[i]; return true; },
                                 hist, bc);
  const int64_t rev = block_count(cnt, [&](int64_t i) {
    return cutu[i] >= 0 && (uint64_t)lb[i] <= cap;
  }, &acc);
  for (int64_t i = threadIdx.x; i < cnt; i += blockDim.x)
    if (cutu[i] >= 0 && (uint64_t)lb[i] <= cap) {
      cu[i] = cutu[i];
      fb[i] = cutu[i];
      cutu[i] = -1;
    }
  if (threadIdx.x == 0 && rev) atomicAdd(nrev, (unsigned long long)rev);
}

// Predictions scattered back to candidate slots: y[oi[j]] = yc[j].
__global__ void k_scatter_y(int64_t n, const int32_t *__restrict__ oi,
                            const float *__restrict__ yc, float *__restrict__ y) {
  const int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (j < n) y[oi[j]] = yc[j];
}

// t = u.q / ||u|| of each pair (FP32; 0 for an invalid user index).
__global__ void k_pair_scores(int64_t npairs, const int32_t *__restrict__ cu,
                              const int32_t *__restrict__ cq, const float *__restrict__ U,
                              const float *__restrict__ Q, int d, float *__restrict__ t) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= npairs) return;
  const int64_t u = cu[i];
  if (u < 0) { t[i] = 0.0f; return; }
  const float *uu = U + u * d, *qq = Q + (int64_t)cq[i] * d;
  float s = 0.0f, nn = 0.0f;
  for (int k = 0; k < d; ++k) {
    s = fmaf(uu[k], qq[k], s);
    nn = fmaf(uu[k], uu[k], nn);
  }
  t[i] = nn > 0.0f ? s / sqrtf(nn) : 0.0f;
}

// t of compacted candidate pairs: x / ||u|| from the screened score x = cx[fi] of
// the pair (the network needs no exact t), else the FP32 product of the rows.
__global__ void k_pair_t(int64_t npairs, const int32_t *__restrict__ fu,
                         const int32_t *__restrict__ fq, const int32_t *__restrict__ fi,
                         const float *__restrict__ cx, const float *__restrict__ unrm,
                         const float *__restrict__ U, const float *__restrict__ Q, int d,
                         float *__restrict__ t) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= npairs) return;
  const int64_t u = fu[i];
  const float x = cx[fi[i]];
  const float nu = unrm[u];
  if (x == x && nu > 0.0f) {
    t[i] = x / nu;
    return;
  }
  const float *uu = U + u * d, *qq = Q + (int64_t)fq[i] * d;
  float s = 0.0f, nn = 0.0f;
  for (int k = 0; k < d; ++k) {
    s = fmaf(uu[k], qq[k], s);
    nn = fmaf(uu[k], uu[k], nn);
  }
  t[i] = nn > 0.0f ? s / sqrtf(nn) : 0.0f;
}

// Per user: R u / ||u|| (64 values) and log ||u||.
__global__ void k_user_features(int64_t n, int d, const float *__restrict__ U,
                                const float *__restrict__ R, float *__restrict__ Xu) {
  const int64_t u = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (u >= n) return;
  const float *uu = U + u * d;
  float nn = 0.0f;
  for (int k = 0; k < d; ++k) nn = fmaf(uu[k], uu[k], nn);
  const float nrm = sqrtf(nn), inv = nrm > 0.0f ? 1.0f / nrm : 0.0f;
  for (int j = 0; j < 64; ++j) {
    float a = 0.0f;
    for (int k = 0; k < d; ++k) a = fmaf(R[j * d + k], uu[k], a);
    Xu[u * 65 + j] = a * inv;
  }
  Xu[u * 65 + 64] = logf(fmaxf(nrm, 1e-30f));
}

rkr_status user_features(const rkr_index *idx, const float *R, float *Xu, cudaStream_t st) {
  k_user_features<<<(unsigned)((idx->n + 127) / 128), 128, 0, st>>>(idx->n, idx->d, idx->U, R,
                                                                     Xu);
  note_launch();
  RKR_CUDA(cudaGetLastError());
  return RKR_OK;
}

rkr_status pair_scores(const rkr_index *idx, const float *Qd, int64_t npairs, const int32_t *cu,
                       const int32_t *cq, float *t, cudaStream_t st) {
  if (npairs <= 0) return RKR_OK;
  k_pair_scores<<<(unsigned)((npairs + 127) / 128), 128, 0, st>>>(npairs, cu, cq, idx->U, Qd,
                                                                   idx->d, t);
  note_launch();
  RKR_CUDA(cudaGetLastError());
  return RKR_OK;
}

static rkr_status query_exact_core(const rkr_index *idx, const QueryCommon &qc, int nq,
                                   const LearnedPrune *lp, int32_t *users_d, int32_t *ranks_d,
                                   rkr_query_stats *stats, cudaStream_t st);

rkr_status run_query_exact(const rkr_index *idx, const QueryCommon &qc, int nq,
                           int32_t *users_d, int32_t *ranks_d, rkr_query_stats *stats,
                           cudaStream_t st) {
  return query_exact_core(idx, qc, nq, nullptr, users_d, ranks_d, stats, st);
}

rkr_status run_query_exact_learned(const rkr_index *idx, const QueryCommon &qc, int nq,
                                   rkr_pruner *pr, const float *Xu, const int32_t *keep_d,
                                   int certify, bool use_table, int32_t *users_d,
                                   int32_t *ranks_d, rkr_query_stats *stats, cudaStream_t st) {
  const LearnedPrune lp{pr, Xu, keep_d, certify, use_table};
  return query_exact_core(idx, qc, nq, &lp, users_d, ranks_d, stats, st);
}

// The learned cut of one chunk: predictions for the candidates still to be
// recounted (nfb of them, compacted), then k_learned_cut per query.
static rkr_status learned_cut(const rkr_index *idx, const QueryCommon &qc, const LearnedPrune *lp,
                              int qa, int qb, int64_t cnt, int64_t nfb, const int64_t *qoff_rel,
                              const uint32_t *cursor, int32_t *cu, const int32_t *cq,
                              const float *cx, int32_t *cu_fb, uint32_t *ccount, int32_t *cutu,
                              int64_t *cut_total, cudaStream_t st) {
  DevBuf b1, b2, b3, b4, b5, b6, b7, b8;
  int32_t *fu, *fq, *fi;
  unsigned long long *cur, *ncut;
  float *tq, *yc, *y;
  RKR_TRY(tmp_alloc(b1, &fu, nfb, st));
  RKR_TRY(tmp_alloc(b2, &fq, nfb, st));
  RKR_TRY(tmp_alloc(b3, &fi, nfb, st));
  RKR_TRY(tmp_alloc(b4, &cur, 1, st));
  RKR_TRY(tmp_alloc(b5, &ncut, 1, st));
  RKR_TRY(tmp_alloc(b6, &tq, nfb, st));
  RKR_TRY(tmp_alloc(b7, &yc, nfb, st));
  RKR_TRY(tmp_alloc(b8, &y, cnt, st));
  RKR_CUDA(cudaMemsetAsync(cur, 0, sizeof(unsigned long long), st));
  RKR_CUDA(cudaMemsetAsync(ncut, 0, sizeof(unsigned long long), st));
  k_compact<<<(unsigned)((cnt + 255) / 256), 256, 0, st>>>(cnt, cu_fb, cq, cur, fu, fq, fi);
  note_launch();
  RKR_CUDA(cudaGetLastError());
  // the network's input t = u.q / ||u||: from the candidate's screened score where
  // it has one (no row is read), else from the rows
  k_pair_t<<<(unsigned)((nfb + 127) / 128), 128, 0, st>>>(nfb, fu, fq, fi, cx, idx->unrm, idx->U,
                                                          qc.Qd, idx->d, tq);
  note_launch();
  RKR_CUDA(cudaGetLastError());
  if (lp->table) {   // one lookup per pair in the user's table
    ProfScope prof("pruner_table", st);
    RKR_TRY(pruner_table_predict(lp->pr, fu, tq, nfb, yc, st));
  } else {
    ProfScope prof("pruner_forward", st);
    RKR_TRY(pruner_forward_gather(lp->pr, lp->Xu, fu, tq, nfb, yc, st));
  }
  k_scatter_y<<<(unsigned)((nfb + 255) / 256), 256, 0, st>>>(nfb, fi, yc, y);
  note_launch();
  // the uncut rule exists for the fallback's sake (n_users = 0 switches it off)
  k_learned_cut<<<qb - qa, filter_threads(cnt, qb - qa), 0, st>>>(qa, qoff_rel, cursor, lp->keep, y, cu_fb, cu, ccount,
                                         cutu, lp->certify ? idx->n : 0, ncut);
  note_launch();
  RKR_CUDA(cudaGetLastError());
  unsigned long long h = 0;
  RKR_CUDA(cudaMemcpyAsync(&h, ncut, sizeof(h), cudaMemcpyDeviceToHost, st));
  RKR_CUDA(cudaStreamSynchronize(st));
  *cut_total += (int64_t)h;
  return RKR_OK;
}

static rkr_status query_exact_core(const rkr_index *idx, const QueryCommon &qc, int nq,
                                   const LearnedPrune *lp, int32_t *users_d, int32_t *ranks_d,
                                   rkr_query_stats *stats, cudaStream_t st) {
  DevBuf bn, bcap;
  int32_t *lstar_d;
  int64_t *ncand_d;
  uint32_t *cap_d;
  RKR_TRY(tmp_alloc(bn, (char **)&ncand_d, plan_bytes(nq), st));
  lstar_d = (int32_t *)(ncand_d + nq);
  RKR_TRY(tmp_alloc(bcap, &cap_d, nq, st));
  DevBuf bw;
  CallWords *words;
  RKR_TRY(words_alloc(bw, &words, st));
  unsigned long long *ties_d = words->ties;
  DevBuf bls;
  unsigned long long *lstat;
  RKR_TRY(tmp_alloc(bls, &lstat, 6, st));   // [5]: candidates still to be recounted
  DevBuf bqs;
  int32_t *qself;
  RKR_TRY(tmp_alloc(bqs, &qself, nq, st));
  RKR_TRY(query_self(idx, qc.Qd, nq, qself, st));
  int64_t fallback = 0, list_fp64 = 0, cut_total = 0;
  double err_ratio = 0.0, err_rel = 0.0;
  int64_t recount_users = 0;   // counted for the caller's statistics alone
  int64_t *const count_users = stats ? &recount_users : nullptr;
  int64_t recount_open = 0, recount_split = 0, revived = 0;
  int64_t prefix_rows = 0, prefix_pruned = 0, canon_rows = 0, canon_theta = 0;
  unsigned long long lstat_host_fb = 0;
  Plan plan;
  double ms_theta = 0.0, ms_res = 0.0, ms_sel = 0.0;
  SpanClock clk(st);
  const int t1 = clk.begin(&ms_theta);
  const Grid grid{qc.xbf,   idx->xg0, idx->xg,       idx->XJU, idx->XJL, idx->nlev_x,
                  idx->XHI, idx->XLO, (uint32_t)idx->m, 1u};
  RKR_TRY(screen_plan(idx, qc, nq, grid, st, lstar_d, cap_d, ncand_d, plan));
  clk.end(t1);
  int wide = 0;
  for (int q = 0; q < nq; ++q) wide += plan.lstar[q] >= idx->nlev_x - 1;
  std::vector<int64_t> qoff(nq + 1, 0);
  for (int q = 0; q < nq; ++q) qoff[q + 1] = qoff[q] + plan.ncand[q];
  std::vector<std::vector<int64_t>> rels;   // per chunk, copied from until the call settles
  StreamGuard guard(st);
  for (auto ch : chunk_queries(plan.ncand, candidate_budget())) {
    int qa = ch.first, qb = ch.second;
    int64_t cnt = qoff[qb] - qoff[qa];
    DevBuf b1, b2, b3, b4, b8, b9;
    int32_t *cu, *cq;
    uint32_t *cursor, *ccount;
    float *cx;
    int64_t *qoff_rel;
    RKR_TRY(tmp_alloc(b9, &cx, cnt, st));
    RKR_CUDA(cudaMemsetAsync(cx, 0xff, sizeof(float) * std::max<int64_t>(cnt, 1), st));  // NaN
    RKR_TRY(tmp_alloc(b1, &cu, cnt, st));
    RKR_TRY(tmp_alloc(b2, &cq, cnt, st));
    RKR_TRY(tmp_alloc(b3, &cursor, nq, st));
    RKR_TRY(tmp_alloc(b4, &ccount, cnt, st));
    RKR_TRY(tmp_alloc(b8, &qoff_rel, nq + 1, st));
    rels.emplace_back(nq + 1, 0);
    std::vector<int64_t> &rel = rels.back();
    for (int q = 0; q <= nq; ++q) rel[q] = qoff[q] - qoff[qa];
    RKR_CUDA(cudaMemcpyAsync(qoff_rel, rel.data(), sizeof(int64_t) * (nq + 1),
                             cudaMemcpyHostToDevice, st));
    RKR_CUDA(cudaMemsetAsync(cursor, 0, sizeof(uint32_t) * nq, st));
    RKR_CUDA(cudaMemsetAsync(cu, 0xff, sizeof(int32_t) * std::max<int64_t>(cnt, 1), st));
    // (the learned cut takes t of a screen's own candidates from their rows)
    const int t2 = clk.begin(&ms_theta);
    RKR_TRY(emit_candidates(idx, qc, qa, qb, grid, plan, lstar_d, cap_d, qoff_rel, cursor, cu, cq,
                            cx, !lp, words, st));
    clk.end(t2);
    const int t3 = clk.begin(&ms_res);
    if (cnt > 0) {
      DevBuf bfb, blb;
      int32_t *cu_fb;
      uint32_t *clb;
      RKR_TRY(tmp_alloc(bfb, &cu_fb, cnt, st));
      RKR_TRY(tmp_alloc(blb, &clb, cnt, st));
      RKR_CUDA(cudaMemsetAsync(lstat, 0, 6 * sizeof(unsigned long long), st));
      {
        const int prof_slot = prof_begin("k_list_rank", st);
        k_list_rank<<<(unsigned)((cnt + 127) / 128), 128, 0, st>>>(
            cnt, cu, cq, cx, qc.Qt.rb3, idx->U, idx->unrm, qc.Qd, idx->Ps, idx->pnrm_s, idx->d,
            idx->xlist, idx->xloff, idx->xlcap, idx->xcoff, idx->xlcnt, idx->xbmax, idx->Ut.rb3, idx->ptile3,
            idx->ptile_bn, tc_gacc(idx->Ut.kp, 1), tc_gcan(idx->d), idx->xg0, idx->xbin, idx->xg,
            idx->ldx, idx->lbin, kListG,
            idx->XLO, idx->XHI, (uint32_t)idx->m, ccount, clb, cu_fb, qself, deep_grid(idx),
            lstat);
        prof_end(prof_slot, st, 0.0);
      }
      note_launch();
      RKR_CUDA(cudaGetLastError());
      {
        const int prof_slot = prof_begin("k_recount_filter", st);
        k_recount_filter<<<qb - qa, filter_threads(cnt, qb - qa), 0, st>>>(qa, qoff_rel, cursor, qc.kq_d, ccount, clb, cu_fb,
                                                         (uint32_t)idx->m);
        prof_end(prof_slot, st, 0.0);
      }
      note_launch();
      RKR_CUDA(cudaGetLastError());
      // candidates that still need the recount, with the rank statistics
      k_count_valid<<<(unsigned)((cnt + 255) / 256), 256, 0, st>>>(cnt, cu_fb, lstat + 5);
      note_launch();
      RKR_CUDA(cudaGetLastError());
      unsigned long long ls[6] = {0, 0, 0, 0, 0, 0};
      RKR_CUDA(cudaMemcpyAsync(ls, lstat, sizeof(ls), cudaMemcpyDeviceToHost, st));
      RKR_CUDA(cudaStreamSynchronize(st));
      canon_theta += (int64_t)ls[4];
      lstat_host_fb = ls[5];
      err_ratio = std::max(err_ratio, (double)u32_float((uint32_t)ls[2]));
      err_rel = std::max(err_rel, (double)u32_float((uint32_t)ls[3]));
      DevBuf bcut;
      int32_t *cutu = nullptr;
      if (lp) {
        RKR_TRY(tmp_alloc(bcut, &cutu, cnt, st));
        RKR_CUDA(cudaMemsetAsync(cutu, 0xff, sizeof(int32_t) * cnt, st));
      }
      if (lp && lstat_host_fb > 0) {  // learned cut of the candidates still to be recounted
        RKR_TRY(learned_cut(idx, qc, lp, qa, qb, cnt, (int64_t)lstat_host_fb, qoff_rel, cursor,
                            cu, cq, cx, cu_fb, ccount, cutu, &cut_total, st));
        lstat_host_fb = 0;
        DevBuf bn4;
        unsigned long long *nfb4;
        RKR_TRY(tmp_alloc(bn4, &nfb4, 1, st));
        RKR_CUDA(cudaMemsetAsync(nfb4, 0, sizeof(unsigned long long), st));
        k_count_valid<<<(unsigned)((cnt + 255) / 256), 256, 0, st>>>(cnt, cu_fb, nfb4);
        note_launch();
        RKR_CUDA(cudaMemcpyAsync(&lstat_host_fb, nfb4, sizeof(unsigned long long),
                                 cudaMemcpyDeviceToHost, st));
        RKR_CUDA(cudaStreamSynchronize(st));
      }
      fallback += (int64_t)lstat_host_fb;
      list_fp64 += (int64_t)ls[1];
      auto recount_open_candidates = [&](unsigned long long h2) -> rkr_status {
        // count intervals for every remaining candidate, then the cap again; only
        // candidates that can still make the k smallest and whose interval is
        // open go on.  The first pass screens with the single BF16 product (a
        // third of the tensor work, wider intervals), the second with the split
        // product on the candidates still open; the exact pass then resolves the
        // undecided items of those that remain.
        for (int pass = tuning().rc_single_first ? 0 : 1; pass < 2 && h2 > 0; ++pass) {
          const bool first = pass == 0 || !tuning().rc_single_first;
          RKR_TRY(recount_candidates(idx, qc, cnt, cu_fb, cq, cx, qself, ccount, clb, nullptr,
                                     st, first ? count_users : nullptr, pass == 0 ? 0 : 1, 0,
                                     &canon_rows));
          if (pass == 1) recount_split += (int64_t)h2;
          {
            const int prof_slot = prof_begin("k_recount_filter", st);
            k_recount_filter<<<qb - qa, filter_threads(cnt, qb - qa), 0, st>>>(qa, qoff_rel, cursor, qc.kq_d, ccount,
                                                     clb, cu_fb, (uint32_t)idx->m);
            prof_end(prof_slot, st, 0.0);
          }
          note_launch();
          k_drop_decided<<<(unsigned)((cnt + 255) / 256), 256, 0, st>>>(cnt, ccount, clb, cu_fb);
          note_launch();
          RKR_CUDA(cudaGetLastError());
          DevBuf bn3;
          unsigned long long *nfb2;
          RKR_TRY(tmp_alloc(bn3, &nfb2, 1, st));
          RKR_CUDA(cudaMemsetAsync(nfb2, 0, sizeof(unsigned long long), st));
          k_count_valid<<<(unsigned)((cnt + 255) / 256), 256, 0, st>>>(cnt, cu_fb, nfb2);
          note_launch();
          RKR_CUDA(cudaMemcpyAsync(&h2, nfb2, sizeof(h2), cudaMemcpyDeviceToHost, st));
          RKR_CUDA(cudaStreamSynchronize(st));
        }
        recount_open += (int64_t)h2;
        if (h2 > 0)
          RKR_TRY(recount_candidates(idx, qc, cnt, cu_fb, cq, cx, qself, ccount, nullptr, ties_d,
                                     st, nullptr, 1, 0, &canon_rows));
        return RKR_OK;
      };
      if (!lp && lstat_host_fb >= (unsigned long long)kGridMinRows)
        RKR_TRY(grid_prune(idx, qc, qa, qb, cnt, qoff_rel, cursor, cq, cx, ccount, clb, cu_fb,
                           &lstat_host_fb, st));
      if (!lp && tuning().rc_prefix > 0 && lstat_host_fb >= (unsigned long long)prefix_min_rows(1))
        RKR_TRY(prefix_prune(idx, qc, qa, qb, cnt, qoff_rel, cursor, cq, cx, qself, ccount, clb, cu_fb,
                             count_users, &lstat_host_fb, &prefix_rows, &prefix_pruned,
                             &canon_rows, st));
      if (lstat_host_fb > 0) RKR_TRY(recount_open_candidates(lstat_host_fb));
      if (lp && lp->certify && cut_total > 0) {
        // exact fallback: cut candidates that could still be among the k best
        DevBuf brv;
        unsigned long long *nrev, hrev = 0;
        RKR_TRY(tmp_alloc(brv, &nrev, 1, st));
        RKR_CUDA(cudaMemsetAsync(nrev, 0, sizeof(unsigned long long), st));
        k_learned_revive<<<qb - qa, 256, 0, st>>>(qa, qoff_rel, cursor, qc.kq_d, ccount, clb,
                                                  cu_fb, cu, cutu, nrev);
        note_launch();
        RKR_CUDA(cudaGetLastError());
        RKR_CUDA(cudaMemcpyAsync(&hrev, nrev, sizeof(hrev), cudaMemcpyDeviceToHost, st));
        RKR_CUDA(cudaStreamSynchronize(st));
        revived += (int64_t)hrev;
        fallback += (int64_t)hrev;
        if (hrev > 0) RKR_TRY(recount_open_candidates(hrev));
      }
    }
    clk.end(t3);
    const int t4 = clk.begin(&ms_sel);
    size_t sm = sizeof(SortEnt) * kMaxK;
    RKR_CUDA(cudaFuncSetAttribute(k_select_exact, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  (int)sm));
    {
      const int prof_slot = prof_begin("k_select_exact", st);
      k_select_exact<<<qb - qa, qb - qa <= sm_count() ? kSelThreadsFew : kSelThreads, sm, st>>>(qa, qoff_rel, cursor, cu, ccount, qc.kq_d,
                                                       qc.out_off_d, users_d, ranks_d,
                                                       &words->select_err,
                                                       (uint32_t)idx->m, user_bits(idx->n));
      prof_end(prof_slot, st, 0.0);
    }
    note_launch();
    RKR_CUDA(cudaGetLastError());
    clk.end(t4);
  }
  CallWords hw;
  RKR_TRY(words_check(words, hw, st));
  guard.settled = true;
  clk.finish();
  const int64_t total = (int64_t)hw.candidates;
  if (stats) {
    stats->pairs = idx->n * (int64_t)nq;
    stats->candidates = total;
    // canonical u.q of list-ranked candidates that needed it, of every recounted
    // row, the near-tie items of the recount and the list entries next to u.q
    stats->fp64_dots = canon_theta + canon_rows + (int64_t)hw.ties[1] + list_fp64;
    stats->near_ties = (int64_t)hw.ties[0];
    stats->recounted = fallback;
    stats->recount_users = recount_users;
    stats->recount_open = recount_open;
    stats->recount_split = recount_split;
    stats->max_rel_screen_err = err_rel;
    stats->max_screen_err_ratio = err_ratio;
    if (lp) stats->candidates = total - cut_total + revived;  // left by the learned cut
    stats->learned_revived = revived;
    stats->prefix_rows = prefix_rows;
    stats->prefix_pruned = prefix_pruned;
    stats->wide_queries = wide;
    stats->deep_queries = (int32_t)plan.deep.size();
    stats->ms_theta = ms_theta;
    stats->ms_resolve = ms_res;
    stats->ms_select = ms_sel;
  }
  return RKR_OK;
}

__global__ void k_count_to_rank(int64_t n, const uint32_t *__restrict__ c,
                                int32_t *__restrict__ r) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i < n) r[i] = (int32_t)(c[i] + 1u);
}

rkr_status run_rank_pairs(const rkr_index *idx, const QueryCommon &qc, int nq, int64_t npairs,
                          const int32_t *cu, const int32_t *cq, int32_t *out_rank,
                          cudaStream_t st) {
  if (npairs <= 0) return RKR_OK;
  DevBuf bq, bc, bl, bf, bs, bt;
  int32_t *qself, *cu_fb;
  uint32_t *ccount, *clb;
  unsigned long long *lstat, *ties;
  RKR_TRY(tmp_alloc(bq, &qself, nq, st));
  RKR_TRY(tmp_alloc(bc, &ccount, npairs, st));
  RKR_TRY(tmp_alloc(bl, &clb, npairs, st));
  RKR_TRY(tmp_alloc(bf, &cu_fb, npairs, st));
  RKR_TRY(tmp_alloc(bs, &lstat, 5, st));
  RKR_TRY(tmp_alloc(bt, &ties, 2, st));
  RKR_CUDA(cudaMemsetAsync(lstat, 0, 5 * sizeof(unsigned long long), st));
  RKR_CUDA(cudaMemsetAsync(ties, 0, 2 * sizeof(unsigned long long), st));
  RKR_TRY(query_self(idx, qc.Qd, nq, qself, st));
  k_list_rank<<<(unsigned)((npairs + 127) / 128), 128, 0, st>>>(
      npairs, cu, cq, nullptr, nullptr, idx->U, idx->unrm, qc.Qd, idx->Ps, idx->pnrm_s, idx->d,
      idx->xlist,
      idx->xloff, idx->xlcap, idx->xcoff, idx->xlcnt, idx->xbmax, idx->Ut.rb3, idx->ptile3,
      idx->ptile_bn, tc_gacc(idx->Ut.kp, 1), tc_gcan(idx->d), idx->xg0, idx->xbin, idx->xg,
      idx->ldx, idx->lbin, kListG, idx->XLO, idx->XHI, (uint32_t)idx->m, ccount, clb, cu_fb, qself,
      deep_grid(idx), lstat);
  note_launch();
  RKR_CUDA(cudaGetLastError());
  unsigned long long ls[2] = {0, 0};
  RKR_CUDA(cudaMemcpyAsync(ls, lstat, sizeof(ls), cudaMemcpyDeviceToHost, st));
  RKR_CUDA(cudaStreamSynchronize(st));
  if (ls[0] > 0)  // pairs below their user's tail list: exact recount
    RKR_TRY(recount_candidates(idx, qc, npairs, cu_fb, cq, nullptr, qself, ccount, nullptr, ties, st));
  k_count_to_rank<<<(unsigned)((npairs + 255) / 256), 256, 0, st>>>(npairs, ccount, out_rank);
  note_launch();
  RKR_CUDA(cudaGetLastError());
  return RKR_OK;
}

}  // namespace rkr
