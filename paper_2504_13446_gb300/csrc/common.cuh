// common.cuh -- shared definitions of the GB300 reverse k-ranks library.
//
// Score arithmetic.  The canonical score s(u,x) is the left-to-right FP64 sum
// of the exact products (double)u[k]*(double)x[k] (the library's reading of
// Def. 1, which fixes no precision).  Bulk work computes cheaper screened
// scores s_hat together with a rigorous bound b such that
// |s_hat - s(u,x)| <= b; a decision is taken from the screen when the bound
// settles it and from canonical FP64 otherwise.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <vector>

#include "rkr.h"

namespace rkr {

// Device memory of the library comes from one stream-ordered pool per device
// that keeps what is freed (its release threshold is unlimited), so index
// builds and query batches reuse the same blocks instead of mapping and
// unmapping tens of GB each time.  rkr_release_cached_memory trims it.
cudaMemPool_t lib_pool();

// Count of device allocations the library has requested (rkr_device_allocations).
void note_alloc();

// Whether this allocation is the one that rkr_set_alloc_fault made the calling thread fail.
bool alloc_fault();

template <class T>
inline cudaError_t pool_malloc_async(T **p, size_t bytes, cudaStream_t st) {
  note_alloc();
  if (alloc_fault()) return cudaErrorMemoryAllocation;
  return cudaMallocFromPoolAsync((void **)p, bytes, lib_pool(), st);
}


constexpr int kMaxD = 256;          // largest supported dimension
constexpr int kMaxLevels = 32;      // rank levels 2^L used by the candidate filter
constexpr int kMaxK = 4096;         // largest k per query

// ------------------------------------------------------------ error state

void set_error(const char *fmt, ...);
rkr_status fail(rkr_status st, const char *fmt, ...);
rkr_status cuda_fail(cudaError_t e, const char *what);

// Count of kernels this library has launched (reported by rkr_kernel_launches).
void note_launch();

// RKR_EUNSUPPORTED unless the current device is sm_103 (GB300).
rkr_status check_device();

// The process-wide tuning (rkr_tuning_set / rkr_autotune), read at launch time.
rkr_tuning tuning();

// Per-kernel device-time accounting, on while rkr_profile_start is in effect:
// CUDA events recorded on the launching stream around a launch.  `work` is the
// launch's algorithmic work (flops of a screen; 0 when not stated).
int prof_begin(const char *name, cudaStream_t st);
void prof_end(int slot, cudaStream_t st, double work);
struct ProfScope {
  int slot;
  cudaStream_t st;
  double work;
  ProfScope(const char *name, cudaStream_t s, double w = 0.0)
      : slot(prof_begin(name, s)), st(s), work(w) {}
  ~ProfScope() { prof_end(slot, st, work); }
};

#define RKR_CUDA(expr)                                            \
  do {                                                            \
    cudaError_t _e = (expr);                                      \
    if (_e != cudaSuccess) return ::rkr::cuda_fail(_e, #expr);    \
  } while (0)

#define RKR_TRY(expr)                                             \
  do {                                                            \
    rkr_status _s = (expr);                                       \
    if (_s != RKR_OK) return _s;                                  \
  } while (0)

// ------------------------------------------------------- canonical scores

// FP64 is scarce on this GPU: a dependent FP64 add or FMA takes 65 cycles, a
// division 590, and a warp's FP64 instruction holds one of the SM's four FP64 units
// for 76 cycles whatever its active lanes (measured).  So hot code decides with
// FP32 bounds and forms canonical scores only for what those leave open.  Rows are read 16 bytes at a time where both allow it: a
// thread per pair touches 32 lines per warp and load either way.

__device__ __forceinline__ bool rows_vec4(const float *a, const float *b, int d) {
  return (d & 3) == 0 && ((((uintptr_t)a) | ((uintptr_t)b)) & 15) == 0;
}

// Calls f(a[k], b[k]) for k = 0 .. d - 1 in order.
template <class F>
__device__ __forceinline__ void for_pairs(const float *__restrict__ a,
                                          const float *__restrict__ b, int d, F &&f) {
  if (rows_vec4(a, b, d)) {
    const float4 *a4 = reinterpret_cast<const float4 *>(a);
    const float4 *b4 = reinterpret_cast<const float4 *>(b);
#pragma unroll 2
    for (int k = 0; k < d >> 2; ++k) {
      const float4 x = a4[k], y = b4[k];
      f(x.x, y.x);
      f(x.y, y.y);
      f(x.z, y.z);
      f(x.w, y.w);
    }
  } else {
    for (int k = 0; k < d; ++k) f(a[k], b[k]);
  }
}

// s(a, b): left-to-right FP64 sum of exact float products (the product of two
// floats is exact in FP64, so one FMA rounds exactly like the addition alone).
__device__ __forceinline__ double canon_dot(const float *__restrict__ a,
                                            const float *__restrict__ b, int d) {
  double acc = 0.0;
  for_pairs(a, b, d, [&](float x, float y) { acc = __fma_rn((double)x, (double)y, acc); });
  return acc;
}

// (double)x of a finite float by integer operations: the conversion instruction
// runs on the FP64 units, four per SM.
__device__ __forceinline__ double exact_double(float x) {
  const bool sub = fabsf(x) < 0x1p-126f;               // a subnormal, scaled to a normal
  const uint32_t b = __float_as_uint(sub ? __fmul_rn(x, 0x1p64f) : x);
  const uint32_t mag = b & 0x7fffffffu;
  const uint32_t bias = sub ? (896u - 64u) << 20 : 896u << 20;
  const uint32_t hi = mag ? (mag >> 3) + bias : 0u;
  return __hiloint2double((int)((b & 0x80000000u) | hi), (int)(b << 29));
}

// Out-of-line copy for rarely taken paths inside unrolled loops.
static __device__ __noinline__ double canon_dot_slow(const float *__restrict__ a,
                                                     const float *__restrict__ b, int d) {
  return canon_dot(a, b, d);
}

// A compensated FP32 dot product (Ogita, Rump and Oishi's Dot2: each product split
// exactly by an FMA, each addition by an error-free two-sum, the low parts summed
// apart): p + s, with |(p + s) - a.b| <= gamma_d^2 sum|a_k b_k| (gamma_d = d u /
// (1 - d u), u = 2^-24).  The canonical sum differs from a.b by at most gamma'_d
// sum|a_k b_k| with the FP64 unit 2^-53.  err bounds |(p + s) - s(a, b)| and the
// rounding of p + s to double, in FP32 rounded up: gamma_d <= g (1 + 2 g) for
// g = d u <= 1/4, and a tiny absolute term covers products in the subnormal range.
// Intrinsics keep the compiler from fusing or reordering the steps.
struct Dot2 {
  float p = 0.0f, s = 0.0f, asum = 0.0f;
  __device__ __forceinline__ void add(float x, float y) {
    const float h = __fmul_rn(x, y);
    const float r = __fmaf_rn(x, y, -h);
    const float t = __fadd_rn(p, h);
    const float z = __fsub_rn(t, p);
    const float e = __fadd_rn(__fsub_rn(p, __fsub_rn(t, z)), __fsub_rn(h, z));
    p = t;
    s = __fadd_rn(s, __fadd_rn(e, r));
    asum = __fadd_ru(asum, fabsf(h));
  }
  // roundings: how many additions a term can pass through (d for one chain)
  __device__ __forceinline__ float err(int roundings) const {
    const float g = (float)roundings * 0x1p-24f;
    const float gam = __fmul_ru(g, __fadd_ru(1.0f, 2.0f * g));
    const float c = __fmaf_ru(gam, gam, __fmul_ru((float)roundings, 0x1.0001p-53f));
    const float e = __fadd_ru(__fmul_ru(c, asum),
                              __fmul_ru(__fadd_ru(fabsf(p), fabsf(s)), 0x1p-52f));
    return __fmul_ru(__fadd_ru(e, (float)roundings * 0x1p-140f), 1.0f + 0x1p-19f);
  }
};

// FP32 upper bound of a Euclidean norm from its FP64 value (the square root of a sum
// of exact squares, up to 2^-44 off): the one definition of these bounds.
__device__ __forceinline__ float norm_up64(double nv) {
  return __double2float_ru(nv * (1.0 + 0x1p-40) + 1e-300);
}

// The same bound, bit for bit, from compensated FP32 sums (all but some 2^-14 of the
// rows need no FP64 operation).  Squares of scaled values (a power of two brings the
// row's largest magnitude near 1) are summed as in Dot2; all terms are non-negative
// and one passes at most 8 + 5 additions here (a lane's eight, five of the warp), so
// that with u = 2^-24 the low parts stay within 14 u of p and the sum p + s within
// 233 u^2 < 2^-40 (relative) of the exact one.
struct SquareSum {
  float p = 0.0f, s = 0.0f;
  __device__ __forceinline__ void two_sum(float h, float low) {
    const float t = __fadd_rn(p, h);
    const float z = __fsub_rn(t, p);
    const float e = __fadd_rn(__fsub_rn(p, __fsub_rn(t, z)), __fsub_rn(h, z));
    p = t;
    s = __fadd_rn(s, __fadd_rn(e, low));
  }
  __device__ __forceinline__ void add(float x) {
    const float h = __fmul_rn(x, x);
    two_sum(h, __fmaf_rn(x, x, -h));
  }
  // over the 32 lanes of a warp
  __device__ __forceinline__ void warp_sum() {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const float p2 = __shfl_xor_sync(0xffffffffu, p, o);
      const float s2 = __shfl_xor_sync(0xffffffffu, s, o);
      two_sum(p2, s2);
    }
  }
  // norm_up64 of sqrt(sum) * unscale; false when these bits do not decide it (also for
  // sums so small that underflow, 2^-140 in all, could matter).  With
  // A = p + s the FP64 form rounds up a T with A < T^2 < A (1 + 2^-38) (its factor
  // 1 + 2^-40 against the 2^-40 above and 2^-44 of its own), so it gives the smallest
  // float r with r^2 > A, unless r^2 lies within A (1 + 2^-38).  A = t + l exactly, and
  // r^2 - t is exact or, a neighbour further off, right in sign and to 2^-24.
  __device__ __forceinline__ bool norm_up(float unscale, float &out) const {
    const float t = __fadd_rn(p, s), l = __fsub_rn(s, __fsub_rn(t, p));
    out = 0.0f;
    if (!(t >= 0x1p-90f)) return false;
    auto over = [&](float r) { return __fsub_rn(__fmaf_rn(r, r, -t), l); };
    const uint32_t r0 = __float_as_uint(__fsqrt_rn(t));
    float r = 0.0f, d = 0.0f;
#pragma unroll
    for (int i = 2; i >= -2; --i) {   // sqrt(A) is within an ulp of the root of t
      const float x = __uint_as_float(r0 + i), e = over(x);
      if (e > 0.0f) {
        r = x;
        d = e;
      }
    }
    out = __fmul_ru(r, unscale);
    return d > __fmul_ru(t, 0x1p-37f);
  }
};

// Power of two that brings mx (a row's largest magnitude) near 1, and its inverse;
// both are normal floats for every mx.
__device__ __forceinline__ void row_scale(float mx, float &scale, float &unscale) {
  int e = (int)(__float_as_uint(mx) >> 23) - 127;   // exponent of mx (-127: zero or subnormal)
  e = max(-126, min(e, 126));
  scale = __uint_as_float((uint32_t)(127 - e) << 23);
  unscale = __uint_as_float((uint32_t)(127 + e) << 23);
}

// Interval [lo, hi] that holds the canonical score s(a, b); everything when a product
// or a sum of the rows leaves the range of float (the ends are then NaN).
__device__ __forceinline__ void dot2_interval(const float *__restrict__ a,
                                              const float *__restrict__ b, int d, double &lo,
                                              double &hi) {
  Dot2 t;
  for_pairs(a, b, d, [&](float x, float y) { t.add(x, y); });
  const double res = (double)t.p + (double)t.s, E = (double)t.err(d);
  lo = res - E;
  hi = res + E;
  if (!(lo <= hi)) {
    lo = -INFINITY;
    hi = INFINITY;
  }
}

// The same rounded outwards to float, without FP64 operations.
__device__ __forceinline__ void dot2_interval_f(const float *__restrict__ a,
                                                const float *__restrict__ b, int d, float &lo,
                                                float &hi) {
  Dot2 t;
  for_pairs(a, b, d, [&](float x, float y) { t.add(x, y); });
  const float E = t.err(d);
  lo = __fsub_rd(__fadd_rd(t.p, t.s), E);
  hi = __fadd_ru(__fadd_ru(t.p, t.s), E);
  if (!(lo <= hi)) {
    lo = -INFINITY;
    hi = INFINITY;
  }
}

// Threshold t_{j+1} (0-based i = j): f_min + i * delta, delta = (f_max - f_min) / (tau - 1),
// each operation rounded to double in that order (Section 4.2, step 2).
__device__ __forceinline__ double thr_at(double fmin, double delta, int i) {
  return __dadd_rn(fmin, __dmul_rn((double)i, delta));
}

// A first guess of #{i : t_i <= theta} for a grid with step delta, from FP32 where
// the step allows it (the callers' comparisons make it exact).  Always in [0, tau]:
// 0 for a NaN, which no comparison moves.
__device__ __forceinline__ int grid_guess(double theta, double fmin, double delta, int tau) {
  const float df = (float)delta;
  if (df > 1e-30f && df < 1e30f) {
    const float x = __fdividef((float)(theta - fmin), df);
    return !(x >= 0.0f) ? 0 : (x >= (float)tau ? tau : (int)x + 1);
  }
  const double x = (theta - fmin) / delta;
  return !(x >= 0.0) ? 0 : (x >= (double)tau ? tau : (int)floor(x) + 1);
}

// j(theta) = #{i in [0, tau) : t_i <= theta}: the 1-based index of the largest
// threshold not above theta (0 when theta < t_1), Section 4.3 step 1.
__device__ __forceinline__ int exact_j(double theta, double fmin, double delta, int tau) {
  int g;
  if (delta > 0.0) {
    g = grid_guess(theta, fmin, delta, tau);
  } else {
    g = theta >= fmin ? tau : 0;
  }
  while (g < tau && thr_at(fmin, delta, g) <= theta) ++g;
  while (g > 0 && thr_at(fmin, delta, g - 1) > theta) --g;
  return g;
}

// Step-3 estimate (Section 4.3): linear in u.q between (t_j, r_up) and (t_{j+1}, r_low).
__device__ __forceinline__ double interp_est(double theta, int j, uint32_t nlo, uint32_t nup,
                                             double fm, double dl, int tau, uint32_t s) {
  double r_up = __dadd_rn(1.0, __ddiv_rn((double)nup, (double)s));
  double r_low = __dadd_rn(1.0, __ddiv_rn((double)nlo, (double)s));
  if (j >= 1 && j <= tau - 1) {
    double tj = thr_at(fm, dl, j - 1);
    double tj1 = thr_at(fm, dl, j);
    double frac = __ddiv_rn(__dsub_rn(theta, tj), __dsub_rn(tj1, tj));
    return __dsub_rn(r_up, __dmul_rn(__dsub_rn(r_up, r_low), frac));
  }
  return r_up;
}

// c(s) = #{i in [0, tau) : t_i < s}: the number of thresholds a score exceeds
// (Alg. 1 counts p in column j when s(u,p) > t_j).
__device__ __forceinline__ int exact_c(double s, double fmin, double delta, int tau) {
  int g;
  if (delta > 0.0) {
    g = grid_guess(s, fmin, delta, tau);
  } else {
    g = s > fmin ? tau : 0;
  }
  while (g < tau && thr_at(fmin, delta, g) < s) ++g;
  while (g > 0 && thr_at(fmin, delta, g - 1) >= s) --g;
  return g;
}

// Per-user data for fast FP32 bin estimates.  For a value x the ideal bin
// coordinate is v = (x - f_min) / delta; t_i <= x iff i <= v.  v is computed
// in FP32 as (x - fmin32) * invd32 with an error of at most err bins (see
// make_binfp), so every integer outside [v - err, v + err] is decided.
struct BinFP {
  float fmin32;
  float invd32;   // 1/delta, or -1 when delta == 0 (degenerate grid)
  float err;      // error bound of v in bins; > 1e6 means "never decide by FP32"
  float pad;
};

// Upper bound of the bin coordinate of x (non-decreasing in x where it is not NaN).
__device__ __forceinline__ float bin_vhi(const BinFP &b, float x) {
  return __fadd_ru(__fmul_ru(__fsub_ru(x, b.fmin32), b.invd32), b.err);
}

// FP32 bin coordinate lower/upper bounds for x in [xlo, xhi].
__device__ __forceinline__ void bin_coord(const BinFP &b, float xlo, float xhi, float &vlo,
                                          float &vhi) {
  vlo = __fsub_rd(__fmul_rd(__fsub_rd(xlo, b.fmin32), b.invd32), b.err);
  vhi = bin_vhi(b, xhi);
}

// Lower end: ceil(v) clamped into [0, tau] (a lower bound of both c and j).
__device__ __forceinline__ int bin_lo(float v, int tau) {
  if (!(v > 0.0f)) return 0;            // also catches NaN
  if (v >= (float)tau) return tau;
  return (int)ceilf(v);
}

// Upper end: floor(v) + 1 clamped into [0, tau] (an upper bound of both c and j).
__device__ __forceinline__ int bin_hi(float v, int tau) {
  if (!(v >= 0.0f)) return v == v ? 0 : tau;
  if (v >= (float)tau) return tau;
  return (int)floorf(v) + 1;
}

// Rigorous interval [jlo, jhi] containing j(x) = #{t_i <= x} and c(x) = #{t_i < x}
// for every x in [xlo, xhi].  jlo == jhi means both are decided and equal.
// fmin is the FP64 grid origin, used only when delta == 0.
__device__ __forceinline__ void bin_interval(const BinFP &b, double fmin, int tau, float xlo,
                                             float xhi, int &jlo, int &jhi) {
  if (b.invd32 < 0.0f) {  // delta == 0: all thresholds equal f_min
    jlo = ((double)xlo > fmin) ? tau : 0;
    jhi = ((double)xhi < fmin) ? 0 : tau;   // (NaN: undecided)
    return;
  }
  if (b.err > 1e6f) { jlo = 0; jhi = tau; return; }
  float vlo, vhi;
  bin_coord(b, xlo, xhi, vlo, vhi);
  jlo = bin_lo(vlo, tau);
  jhi = bin_hi(vhi, tau);
}

// bin_interval with an error that follows the values: the FP32 coordinate
// (v - f)(1/dx), f = fl(g0), taken with directed roundings, is within
// e(v) = (|v - f| 2^-21 + |g0| 2^-23) / dx of (v - g0) / dx: the roundings of f, of
// 1/dx, of the difference and of the product add up to less than
// |g0| 2^-24 / dx + |v - f| 2^-21.6 / dx.  (1/dx <= invd32 (1 + 2^-22), since invd32
// is 1/dx rounded to nearest twice, and |g0| <= |f| (1 + 2^-23); both factors are
// formed in FP32 rounding up.)  Valid for every v, whatever range err was made
// for; usable() is false for grids without a usable step.
struct TightBins {
  float f, inv, e0, e1;
  bool ok;
  __device__ __forceinline__ explicit TightBins(const BinFP &b) {
    f = b.fmin32;
    inv = b.invd32;
    ok = b.invd32 > 0.0f && b.err <= 1e6f;
    const float inv_up = __fmul_ru(b.invd32, 1.0f + 0x1p-22f);
    e1 = __fmul_ru(inv_up, 0x1p-21f * (1.0f + 0x1p-20f));
    e0 = __fadd_ru(__fmul_ru(__fmul_ru(fabsf(b.fmin32), (1.0f + 0x1p-23f) * 0x1p-23f), inv_up),
                   0x1p-30f);
  }
  __device__ __forceinline__ bool usable() const { return ok; }
  // lower bound of #{x_j <= v} (and of #{x_j < v}) over G columns
  __device__ __forceinline__ int lo(float v, int G) const {
    const float a = __fsub_rd(v, f);
    const float e = __fmaf_ru(fmaxf(fabsf(a), fabsf(__fsub_ru(v, f))), e1, e0);
    return bin_lo(__fsub_rd(__fmul_rd(a, inv), e), G);
  }
  // upper bound of the same
  __device__ __forceinline__ int hi(float v, int G) const {
    const float a = __fsub_ru(v, f);
    const float e = __fmaf_ru(fmaxf(fabsf(a), fabsf(__fsub_rd(v, f))), e1, e0);
    return bin_hi(__fadd_ru(__fmul_ru(a, inv), e), G);
  }
};

// FP32 screen bound: |fma-chain(u,x) - s(u,x)| <= cfac * |u| * |x| with
// cfac = ((d + 4) 2^-24 + d 2^-53 + 2^-40)(1 + 2^-20); nu, nx are FP32 upper
// bounds of the Euclidean norms.  The FMA chain rounds once per step, each
// partial sum is at most sum_k |u_k x_k| <= |u||x| (Cauchy-Schwarz); the extra
// terms cover the canonical sum's own rounding and the rounding of s_hat -+ b.
__host__ __device__ __forceinline__ float screen_cfac(int d) {
  double c = ((double)(d + 4) * 0x1p-24 + (double)d * 0x1p-53 + 0x1p-40) * (1.0 + 0x1p-20);
  return (float)c * (1.0f + 0x1p-20f);
}

__device__ __forceinline__ float screen_bound(float cfac, float nu, float nx) {
  return __fadd_ru(__fmul_ru(__fmul_ru(cfac, nu), nx), 1e-30f);
}

// Per-query user subsets as bitmaps: word q * words + u / 32, bit u % 32.  A null
// bitmap means every user belongs to every query.
__device__ __forceinline__ bool in_subset(const uint32_t *__restrict__ member, int64_t words,
                                          int64_t q, int64_t u) {
  return !member || ((member[q * words + (u >> 5)] >> (u & 31)) & 1u);
}

// Level boundaries: level L holds counts N <= B_L = scale * (2^L - 1).
__host__ __device__ __forceinline__ uint64_t level_bound(int L, uint32_t scale) {
  return (uint64_t)scale * (((uint64_t)1 << L) - 1);
}

// Float with the given bit pattern (host and device).
__host__ __device__ __forceinline__ float u32_float(uint32_t b) {
  union {
    uint32_t u;
    float f;
  } x;
  x.u = b;
  return x.f;
}

// ------------------------------------------------------- host helpers

// A stream-ordered temporary from the library pool, freed when it goes out of scope.
struct DevBuf {
  void *p = nullptr;
  cudaStream_t st = nullptr;
  ~DevBuf() {
    if (p) cudaFreeAsync(p, st);
  }
};

// Waits for a stream when a call ends before it has done so itself (settled): on an
// error, kernels and copies that use the caller's arrays or the call's own host
// vectors may still be queued.  Declared after those vectors.
struct StreamGuard {
  cudaStream_t st;
  bool settled = false;
  explicit StreamGuard(cudaStream_t s) : st(s) {}
  ~StreamGuard() {
    if (!settled) cudaStreamSynchronize(st);
  }
  StreamGuard(const StreamGuard &) = delete;
  StreamGuard &operator=(const StreamGuard &) = delete;
};

template <class T>
inline rkr_status tmp_alloc(DevBuf &b, T **out, size_t count, cudaStream_t st) {
  if (count == 0) count = 1;
  cudaError_t e = pool_malloc_async(&b.p, count * sizeof(T), st);
  if (e != cudaSuccess) {
    cudaGetLastError();
    b.p = nullptr;
    return fail(RKR_ENOMEM, "device allocation of %zu bytes failed", count * sizeof(T));
  }
  b.st = st;
  *out = (T *)b.p;
  return RKR_OK;
}

// Device times of stretches of one call: events recorded as the stretches begin and
// end, read once by finish() after the call's own synchronization (no waiting in
// between).
struct SpanClock {
  struct Span {
    cudaEvent_t a, b;
    double *acc;   // milliseconds are added here
  };
  cudaStream_t st;
  std::vector<Span> spans;
  explicit SpanClock(cudaStream_t s) : st(s) {}
  int begin(double *acc) {
    Span x{nullptr, nullptr, acc};
    if (cudaEventCreate(&x.a) != cudaSuccess || cudaEventCreate(&x.b) != cudaSuccess)
      cudaGetLastError();
    spans.push_back(x);
    if (x.a) cudaEventRecord(x.a, st);
    return (int)spans.size() - 1;
  }
  void end(int i) {
    if (spans[i].b) cudaEventRecord(spans[i].b, st);
  }
  void finish() {   // the stream has been synchronized
    for (Span &x : spans) {
      float ms = 0.0f;
      if (x.a && x.b && cudaEventElapsedTime(&ms, x.a, x.b) == cudaSuccess) *x.acc += ms;
      else cudaGetLastError();
    }
  }
  ~SpanClock() {
    for (Span &x : spans) {
      if (x.a) cudaEventDestroy(x.a);
      if (x.b) cudaEventDestroy(x.b);
    }
  }
  SpanClock(const SpanClock &) = delete;
  SpanClock &operator=(const SpanClock &) = delete;
};

// Order-preserving key of a non-negative double.
__device__ __forceinline__ uint64_t dkey(double x) { return (uint64_t)__double_as_longlong(x); }

}  // namespace rkr
