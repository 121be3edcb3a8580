// tc_screen.cuh -- persistent tcgen05 screen kernel with a pluggable epilogue.
//
// Work is a list of units; a unit is a rectangle of tiles [rb0, rb1) x [ct0, ct1)
// (row blocks of 128 users, column tiles of BN items or queries), walked
// row-major.  Row-owned units (one row block, all columns) keep per-user
// epilogue state in the CTA; column-owned units (one column tile, a range of
// row blocks) keep per-column state.
//
// Epi must provide (all called by the epilogue threads, 32 * epi_warps<Epi>() of
// them, const members):
//   struct Thread;                                    per-thread state
//   static constexpr size_t kSmem;                    bytes of epilogue scratch
//   void unit_begin(char *S, const Unit &u, int et, Thread &)   et = 0..threads-1
//   void tile_begin(char *S, int rb, int ct, int r, int h, Thread &)
//   void chunk(char *S, int rb, int ct, int r, int col, uint32_t tm, const float (&v)[32], Thread &)
//   void tile_end(char *S, int rb, int ct, int r, int h, Thread &)
//   void unit_end(char *S, const Unit &u, int et, Thread &)
// r is the accumulator row (0..127), h the column group, col the first of the
// 32 columns of the chunk within the tile.  Named barrier 1 (the epilogue threads)
// is available to unit_begin/unit_end and tile_begin/tile_end as tc::epi_sync<W>(),
// W the epilogue's warps.
#pragma once

#include "tc.cuh"

namespace rkr {
namespace tc {

struct Unit {
  int rb0, rb1, ct0, ct1;
  int slice = 0;    // K mode: the K slice
};

// How units are formed: ROW = one row block each; COL = one column tile and
// one of `parts` slices of the row blocks; K = one tile and one of `parts` slices
// of K, `kparts` chunks each (products with few tiles and a long K, single-CTA
// kernel and one segment only; the epilogue keeps the slices apart).
struct Schedule {
  int mode;       // 0 ROW, 1 COL, 2 K
  int nrb, nct;   // row blocks, column tiles
  int parts;      // COL: row-block slices per column tile; K: slices of K
  int nunits;
  int kparts = 0; // K: chunks per slice
};

__device__ __forceinline__ Unit unit_of(const Schedule &s, int i) {
  Unit u;
  if (s.mode == 0) {
    u.rb0 = i; u.rb1 = i + 1; u.ct0 = 0; u.ct1 = s.nct;
  } else if (s.mode == 2) {
    const int tile = i / s.parts;
    u.slice = i - tile * s.parts;
    u.rb0 = tile / s.nct; u.rb1 = u.rb0 + 1;
    u.ct0 = tile - u.rb0 * s.nct; u.ct1 = u.ct0 + 1;
  } else {
    int ct = i / s.parts, part = i - ct * s.parts;
    u.ct0 = ct; u.ct1 = ct + 1;
    u.rb0 = (int)((int64_t)s.nrb * part / s.parts);
    u.rb1 = (int)((int64_t)s.nrb * (part + 1) / s.parts);
  }
  return u;
}

// The i-th column tile of [ct0, ct1): in order, or (interleaved) from both ends in
// turn.
template <bool INTERLEAVE>
__device__ __forceinline__ int tile_at(int i, int ct0, int ct1) {
  if (!INTERLEAVE) return i;
  const int j = i - ct0;
  return j & 1 ? ct1 - 1 - (j >> 1) : ct0 + (j >> 1);
}
// The tile after `ct` in that order over nct tiles (nct or -1 past the last one).
template <bool INTERLEAVE>
__device__ __forceinline__ int tile_after(int ct, int nct) {
  if (!INTERLEAVE) return ct + 1;
  if (2 * ct == nct - 1 || 2 * ct == nct) return -1;
  return 2 * ct < nct ? nct - 1 - ct : nct - ct;
}

// Whether a screen takes its column tiles from both ends in turn: where the item
// side is sorted by norm, the epilogue's work falls from the first tile to the last,
// and a heavy tile's epilogue then overlaps a light tile's MMAs.  Taken where it
// pays: the list screen of long rows, 98.3 -> 93.1 ms (1M x 100k x 200); the extremes
// 30.1 -> 32.5 (they want the large norms first), the counting screens 3 to 9 % slower.
template <class Epi, class = void>
struct EpiInterleave {
  static constexpr bool value = false;
};
template <class Epi>
struct EpiInterleave<Epi, decltype((void)Epi::kInterleave)> {
  static constexpr bool value = Epi::kInterleave;
};

template <int WARPS>
__device__ __forceinline__ void epi_sync() {
  asm volatile("bar.sync 1, %0;" ::"n"(32 * WARPS) : "memory");
}

// Barrier of the epilogue threads that also ORs a predicate over them, so
// that every epilogue warp takes the same decision at the end of a unit (a warp
// that gave up a bounded wait and one that did not would otherwise disagree on
// the number of barriers still to come).
template <int WARPS>
__device__ __forceinline__ bool epi_vote_any(bool p) {
  uint32_t r;
  asm volatile(
      "{\n .reg .pred a, b;\n setp.ne.u32 a, %1, 0;\n"
      " barrier.red.or.pred b, 1, %2, a;\n selp.u32 %0, 1, 0, b;\n}\n"
      : "=r"(r)
      : "r"((uint32_t)p), "n"(32 * WARPS)
      : "memory");
  return r != 0;
}

// K chunks of a tile in the order they are multiplied: a counter over the chunks
// of `nseg` segments (no division: the issue loops run once per chunk and are on
// the critical path of the MMAs).
struct ChunkWalk {
  int c = 0, g = 0;   // chunk within the segment, segment
  __device__ __forceinline__ void next(int kchunks) {
    if (++c == kchunks) {
      c = 0;
      ++g;
    }
  }
};

// Position in a ring of STAGES pipeline stages and the phase parity of its pass.
template <int STAGES>
struct Ring {
  uint32_t s = 0, ph = 0;
  __device__ __forceinline__ void next() {
    if (++s == (uint32_t)STAGES) {
      s = 0;
      ph ^= 1;
    }
  }
};

// MMA issue for one accumulator tile (whole warp, converged).  The warp walks the
// chunk loop together and one elected lane issues, so that descriptors and
// addresses live in uniform registers; the next stage's barrier is looked at
// before this stage's MMAs are issued, which hides its latency.  Measured per
// 64-wide chunk of a 128 x 256 tile (four MMAs, 516 cycles of tensor pipe): one
// lane in a divergent branch with a division per chunk 920 cycles, this form 570.
// Returns false when a bounded wait gave up.
template <int STAGES, uint32_t kStageBytes, uint32_t kABytes, class Issue, class Free>
__device__ __forceinline__ bool mma_tile(const Operands &op, int nk, uint64_t *full,
                                         uint64_t desc0, Ring<STAGES> &ring, bool &ready,
                                         Issue &&issue, Free &&release) {
  const int last = op.ksteps - (op.kchunks - 1) * 4;   // MMA steps of a segment's last chunk
  int c = 0;
  for (int kc = 0; kc < nk; ++kc) {
    if (!ready && !mbar_wait_warp(&full[ring.s], ring.ph)) return false;
    const uint32_t s = ring.s;
    ring.next();
    ready = mbar_test_warp(&full[ring.s], ring.ph);
    tc_fence_after();
    const uint64_t da = desc0 + (uint64_t)(s * (kStageBytes >> 4));
    const uint64_t db = da + (kABytes >> 4);
    const int steps = ++c == op.kchunks ? last : 4;
    if (c == op.kchunks) c = 0;
    if (elect_one()) {
#pragma unroll
      for (int k = 0; k < 4; ++k)
        if (k < steps) issue(da + 2 * k, db + 2 * k, (kc | k) != 0 ? 1u : 0u);
      release(s, kc == nk - 1);
    }
    __syncwarp();
  }
  return true;
}

// Whether the epilogue's chunk() reads TMEM again (then a tile's accumulator is
// released only after its last chunk; otherwise right after its last load).
template <class Epi, class = void>
struct EpiReloads {
  static constexpr bool value = false;
};
template <class Epi>
struct EpiReloads<Epi, decltype((void)Epi::kReloads)> {
  static constexpr bool value = Epi::kReloads;
};

// This thread's columns of an accumulator row (TMEM row address trow), handed to
// the epilogue as chunks of 32.  With 8 warps a load brings 64 columns (one wait
// for two chunks); with 16, registers allow 32 and other warps cover the wait.
// `release` frees the accumulator once nothing will read it again.
template <int BN, class Epi, class Free>
__device__ __forceinline__ void epi_tile_columns(const Epi &epi, char *S, int rb, int ct, int r,
                                                 int group, uint32_t trow,
                                                 typename Epi::Thread &ts, Free &&release) {
  constexpr int kCols = BN / (epi_warps<Epi>() / 4);   // columns of this thread
  if constexpr (epi_warps<Epi>() == 8) {
#pragma unroll 1
    for (int cc = 0; cc < kCols; cc += 64) {
      const int col = group * kCols + cc;
      float v[64];
      tmem_ld64(trow + col, v);
      if (!EpiReloads<Epi>::value && cc + 64 >= kCols) release();
      epi.chunk(S, rb, ct, r, col, trow + (uint32_t)col,
                *reinterpret_cast<const float(*)[32]>(v), ts);
      epi.chunk(S, rb, ct, r, col + 32, trow + (uint32_t)(col + 32),
                *reinterpret_cast<const float(*)[32]>(v + 32), ts);
    }
  } else {
#pragma unroll 1
    for (int cc = 0; cc < kCols; cc += 32) {
      const int col = group * kCols + cc;
      float v[32];
      tmem_ld32(trow + col, v);
      if (!EpiReloads<Epi>::value && cc + 32 >= kCols) release();
      epi.chunk(S, rb, ct, r, col, trow + (uint32_t)col, v, ts);
    }
  }
  if (EpiReloads<Epi>::value) release();
}

template <int BN>
struct Layout {
  static_assert(BN == 128 || BN == 256, "column tiles of 128 or 256");
  static constexpr uint32_t kA = BM * KCH * 2;      // 16 KB
  static constexpr uint32_t kB = BN * KCH * 2;
  static constexpr uint32_t kStage = kA + kB;
};

template <int BN, int STAGES, class Epi>
__global__ void __launch_bounds__(screen_threads<Epi>(), 1)
    k_screen(const __grid_constant__ CUtensorMap mAh, const __grid_constant__ CUtensorMap mAl,
             const __grid_constant__ CUtensorMap mBh, const __grid_constant__ CUtensorMap mBl,
             Operands op, Schedule sch, Epi epi, int *err) {
  using L = Layout<BN>;
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  // 1024-byte alignment for the swizzled tiles
  unsigned char *base = (unsigned char *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  unsigned char *stages = base;
  uint64_t *full = (uint64_t *)(stages + (size_t)STAGES * L::kStage);
  uint64_t *empty = full + STAGES;
  uint64_t *acc_full = empty + STAGES;
  uint64_t *acc_empty = acc_full + 2;
  uint64_t *drain = acc_empty + 2;
  uint32_t *tmem_slot = (uint32_t *)(drain + 1);
  char *escratch = (char *)(tmem_slot + 4);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int nseg = op.split ? 3 : 1;
  const int nk = op.kchunks * nseg;
  constexpr uint32_t kTmemCols = 2 * BN;

  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&acc_full[b], 1);
      mbar_init(&acc_empty[b], epi_warps<Epi>());
    }
    mbar_init(drain, 1);
    fence_barrier_init();
  }
  if (warp == 1) tmem_alloc(tmem_slot, kTmemCols);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  bool failed = false;

  if (warp == 0) {
    // ---------------------------------------------------------------- TMA
    if (lane == 0) {
      prefetch_map(&mAh); prefetch_map(&mBh);
      if (op.split) { prefetch_map(&mAl); prefetch_map(&mBl); }
      uint32_t it = 0;
      Ring<STAGES> ring;
      const int kstep = op.fp8 ? 2 * KCH : KCH;  // elements of 128 bytes
      for (int ui = blockIdx.x; ui < sch.nunits && !failed; ui += gridDim.x) {
        Unit u = unit_of(sch, ui);
        const int k0 = u.slice * sch.kparts;   // first chunk (K mode), the slice's chunks
        const int uk = sch.mode == 2 ? min(sch.kparts, nk - k0) : nk;
        for (int rb = u.rb0; rb < u.rb1 && !failed; ++rb)
          for (int i = u.ct0; i < u.ct1 && !failed; ++i) {
            const int ct = tile_at<EpiInterleave<Epi>::value>(i, u.ct0, u.ct1);
            ChunkWalk w;
            for (int kc = 0; kc < uk; ++kc, ++it) {
              const uint32_t s = ring.s;
              if (!mbar_wait(&empty[s], ring.ph ^ 1, kWaitLimit, true)) { failed = true; break; }
              unsigned char *sa = stages + (size_t)s * L::kStage;
              unsigned char *sb = sa + L::kA;
              mbar_expect_tx(&full[s], L::kStage);
              // split order: hi.lo, lo.hi, then hi.hi (small terms first)
              const bool alo = op.split && w.g == 1, blo = op.split && w.g == 0;
              const int kx = (k0 + w.c) * kstep;
              tma_load_2d(sa, alo ? &mAl : &mAh, kx, rb * BM, &full[s]);
              tma_load_2d(sb, blo ? &mBl : &mBh, kx, ct * BN, &full[s]);
              w.next(op.kchunks);
              ring.next();
            }
          }
      }
      if (failed) {
        atomicExch(err, 1);
        // let every load already issued land before the CTA can exit
        for (uint32_t j = (it > STAGES ? it - STAGES : 0); j < it; ++j)
          mbar_wait(&full[j % STAGES], (j / STAGES) & 1);
      }
    }
  } else if (warp == 1) {
    // ---------------------------------------------------------------- MMA
    const uint32_t idesc = op.fp8 ? idesc_e4m3(BM, BN) : idesc_bf16(BM, BN);
    const uint64_t desc0 = sw128_desc(smem_u32(stages));
    Ring<STAGES> ring;
    bool ready = false;
    uint32_t t = 0;
    for (int ui = blockIdx.x; ui < sch.nunits && !failed; ui += gridDim.x) {
      Unit u = unit_of(sch, ui);
      const int uk = sch.mode == 2 ? min(sch.kparts, nk - u.slice * sch.kparts) : nk;
      for (int rb = u.rb0; rb < u.rb1 && !failed; ++rb)
        for (int ct = u.ct0; ct < u.ct1 && !failed; ++ct, ++t) {
          const int b = t & 1;
          const uint32_t aph = (t >> 1) & 1;
          if (!mbar_wait_warp(&acc_empty[b], aph ^ 1, kWaitLimit, true)) { failed = true; break; }
          tc_fence_after();
          const uint32_t dt = tmem + (uint32_t)(b * BN);
          failed = !mma_tile<STAGES, L::kStage, L::kA>(
              op, uk, full, desc0, ring, ready,
              [&](uint64_t da, uint64_t db, uint32_t acc) {
                if (op.fp8) umma_e4m3(dt, da, db, idesc, acc);
                else umma_bf16(dt, da, db, idesc, acc);
              },
              [&](uint32_t s, bool last) {
                umma_commit(&empty[s]);
                if (last) umma_commit(&acc_full[b]);
              });
        }
    }
    if (elect_one()) {
      if (failed) atomicExch(err, 2);
      // all MMAs issued by this warp complete before the CTA releases TMEM
      umma_commit(drain);
      mbar_wait(drain, 0);
    }
    __syncwarp();
  } else {
    // ----------------------------------------------------------- epilogue
    constexpr int EW = epi_warps<Epi>();
    const int e = warp - 2;                 // 0 .. EW - 1
    const int et = threadIdx.x - 64;        // 0 .. 32 EW - 1
    const int quarter = warp & 3;
    const int group = e >> 2;               // column group
    const int r = quarter * 32 + lane;      // accumulator row (user within the block)
    uint32_t t = 0;
    typename Epi::Thread ts;
    for (int ui = blockIdx.x; ui < sch.nunits && !failed; ui += gridDim.x) {
      Unit u = unit_of(sch, ui);
      epi.unit_begin(escratch, u, et, ts);
      epi_sync<EW>();
      for (int rb = u.rb0; rb < u.rb1; ++rb)
        for (int i = u.ct0; i < u.ct1; ++i, ++t) {
          const int ct = tile_at<EpiInterleave<Epi>::value>(i, u.ct0, u.ct1);
          const int b = t & 1;
          const uint32_t aph = (t >> 1) & 1;
          // a warp that gave up goes through the rest of the unit without waiting or
          // reading, so that every warp passes the same barriers (the vote below)
          if (!failed && !mbar_wait_warp(&acc_full[b], aph, op.epi_wait)) failed = true;
          tc_fence_after();
          epi.tile_begin(escratch, rb, ct, r, group, ts);
          const uint32_t trow = tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(b * BN);
          if (!failed)
            epi_tile_columns<BN>(epi, escratch, rb, ct, r, group, trow, ts, [&]() {
              tc_fence_before();
              __syncwarp();
              if (lane == 0) mbar_arrive(&acc_empty[b]);
            });
          epi.tile_end(escratch, rb, ct, r, group, ts);
        }
      failed = epi_vote_any<EW>(failed);
      if (!failed) epi.unit_end(escratch, u, et, ts);
      epi_sync<EW>();
    }
    if (failed && lane == 0) atomicExch(err, 3);
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 1) {
    __syncwarp();
    tmem_dealloc(tmem, kTmemCols);
  }
}

// Stages of the single-CTA and multicast forms that fit beside the epilogue's
// scratch (at most 4).
template <int BN, class Epi>
constexpr int stages1() {
  constexpr size_t avail = 232448 - 1024 - 16 - 8 * 13 - Epi::kSmem;
  constexpr int s = (int)(avail / Layout<BN>::kStage);
  return s > 4 ? 4 : s;
}

template <int BN, int STAGES, class Epi>
constexpr size_t screen_smem_bytes() {
  return 1024 + (size_t)STAGES * Layout<BN>::kStage + 8 * (2 * STAGES + 5) + 16 + Epi::kSmem;
}

}  // namespace tc
}  // namespace rkr
