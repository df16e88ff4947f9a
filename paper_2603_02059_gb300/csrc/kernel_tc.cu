// kernel_tc.cu -- the tensor-core path: tcgen05 Gram tiles fed by TMA (Algorithm 1,
// "Symmetric Batched GeMM", with the norm identity of Eq. 4), fused with the
// trajectory window of Eq. 2, the exclusion mask and the per-row top-k
// (Algorithm 1, kNN step). The N x N snapshot matrix never leaves the chip.
//
// Precision forms. BF16: G = <bf16(x_a), bf16(x_b)>. Split-BF16: every centred
// value is written as x = hi + lo with hi = bf16(x), lo = bf16(x - hi), and
//     G = <hi_a, hi_b> + <hi_a, lo_b> + <lo_a, hi_b>
// (the lo.lo term, about 2^-16 of |x_a||x_b|, is dropped), accumulated in FP32
// in tensor memory. The day norms and window sums stay FP64 (kernels_aux.cu).
//
// Operands are the grouped BF16 copies of the operand preparation (kernels_aux.cu):
// per 64 K entries, 63 permuted grid points and one correction entry that makes the
// accumulator hold G - groups c_a c_b (small for close pairs); the epilogue adds
// groups c_a c_b back in FP32.
//
// One persistent CTA per SM, warp-specialised:
//   warp 0   TMA producer: A (128 strip rows) and B (256 tile columns) K-chunks of
//            32 elements into a ring of shared-memory stages (hi and lo copies);
//   warp 1   tcgen05.mma issuer into one of two 128 x 256 FP32 accumulators in
//            TMEM (512 columns). The K range of a tile is cut into segments
//            (8192 elements by default) that accumulate afresh: the tensor cores never
//            accumulate more than one segment of products per output, which bounds the
//            error of their accumulation however large D is. A tile's first segment goes
//            to one accumulator and stays there as its running total; every other one
//            goes to the other accumulator, from where the epilogue adds it to the total
//            in FP32 on the CUDA cores. The next tile takes them the other way round, so
//            its first segment multiplies while the total is scanned;
//   warps 2-  epilogue, in one or two groups of four warps (two split a tile's columns):
//            each thread owns one accumulator row (TMEM lane), pulls 32 columns at a
//            time with tcgen05.ld, stages them beside the L-1 columns carried from the
//            previous chunk, sums each output's window down the diagonal, masks the
//            exclusion zone, and appends the distances within the row's bound to the
//            row's candidate list (row side) and, beyond the strip's own block, those
//            within a column's bound to the column's list (column side), so each
//            unordered pair is evaluated once (epilogue.cuh).
// Work units (a strip and a range of columns, or a band unit that only seeds the
// per-row bounds) are handed out dynamically; a unit may serve several series that
// share its Gram tiles (several trajectory lengths of one record).
// Every wait is bounded (globaltimer); a wait that runs out records a timeout
// in the status word, the CTA (with the other one of its pair) drains its copies and
// MMAs, frees TMEM and returns.
#include <cuda.h>
#include <cuda_runtime.h>
#include <math_constants.h>

#include "epilogue.cuh"
#include "internal.h"
#include "tc_ptx.cuh"

namespace traknn {
namespace {

constexpr int BM = kTileRows;  // accumulator rows (TMEM lanes)
constexpr int BN = kTileCols;  // accumulator columns per tile (256)
constexpr int KC = 32;         // K elements per stage (64 B rows, 64-B swizzle)
constexpr int kEpiThreads = 128;  // one epilogue group: one thread per accumulator row
// Threads of a CTA: warp 0 producer, warp 1 MMA issuer, G epilogue groups of four
// warps. With G = 2 group g reads the columns [g 128, (g+1) 128) of every tile, so that
// twice as many warps hide the epilogue's latencies when it, not the contraction, sets
// the pace.
__host__ __device__ constexpr int kThreadsG(int G) { return 64 + kEpiThreads * G; }
// Pitch of the Gram chunk buffer: 32 columns plus the L-1 carried ones, made odd
// so that the diagonal reads of 32 consecutive rows hit 32 different banks. Without
// windows (every L = 1) a row only holds its own distances: 16-byte aligned rows whose 16-byte
// accesses by eight consecutive lanes hit different banks.
__host__ __device__ constexpr int chunk_pitch(int L, bool win) {
  return !win ? 36 : 32 + (L - 1) + (((L - 1) % 2 == 0) ? 1 : 0);
}
constexpr uint32_t kTileA = BM * KC * 2;  // bytes of one A operand tile
constexpr uint32_t kTileB = BN * KC * 2;  // bytes of one B operand tile
constexpr uint32_t kIdesc = ptx::idesc_bf16_f32(BM, BN);
constexpr uint32_t kIdescPair = ptx::idesc_bf16_f32(2 * BM, BN);
constexpr int kMaxStages = 8;
constexpr size_t kSmemLimit = 232448;  // 227 KB opt-in per block

// Shared memory of one epilogue group: Gram chunk with carried columns, W, row bounds
// and correction values of a tile, column-side counters (two chunks), a tile's finite columns.
__host__ __device__ constexpr size_t group_bytes(int L) {
  return (size_t)BM * chunk_pitch(L, L > 1) * 4 + 3 * BN * 4 + 64 * 4 + BN / 8;
}

struct TcParams {
  TcArgs a;
  TcWork w;
  int nstages;
  int split;
  uint32_t stage_bytes;
  int seg_kb;  // K blocks (of KC elements) per accumulation segment
  SeriesTable sr;
};


struct Ctl {
  volatile int* abort;
  int* err;
  unsigned long long limit_ns;
  uint32_t peer_abort;  // the abort flag of the pair's other CTA (0: a single CTA)
};

// A wait has run out: records the timeout and raises the abort flags.
__device__ __forceinline__ void give_up(const Ctl& c) {
  atomicCAS(c.err, 0, kErrTimeout);
  *c.abort = 1;
  if (c.peer_abort) ptx::st_remote_u32(c.peer_abort, 1u);
}

// Bounded wait on an mbarrier phase. Records a timeout and raises the CTA's abort
// flag (and that of the pair's other CTA, whose roles would wait for this one's) when the
// limit runs out; gives up early when another role aborted.
// kCluster: what the other CTA of a pair wrote before it arrived is visible afterwards.
template <bool kCluster = false>
__device__ __forceinline__ bool wait_bounded(uint32_t bar, uint32_t parity, const Ctl& c,
                                             bool honor_abort = true) {
  auto ready = [&]() {
    return kCluster ? ptx::mbar_try_wait_cluster(bar, parity) : ptx::mbar_try_wait(bar, parity);
  };
  if (ready()) return true;
  const uint64_t t0 = ptx::globaltimer();
  for (;;) {
    if (ready()) return true;
    if (honor_abort && *c.abort) return false;
    if (ptx::globaltimer() - t0 > c.limit_ns) {
      give_up(c);
      return false;
    }
  }
}

constexpr int kQueue = 4;  // depth of the per-CTA unit queue

// G: epilogue groups; kWin: some series of the call has L > 1 (windows are summed); kBand:
// the band pre-pass (bounds only, no lists); kLarge: k > 32 in the band pass (two minima
// per group), k > 40 in the main pass (128 shared minima); one epilogue group only.
//
// kPair (main pass, one epilogue group): clusters of two CTAs work as one on units of two
// neighbouring strips. Each CTA loads its own strip's rows and half of a tile's columns
// (128) and computes its strip's 128 x 256 outputs with both halves (cta_group::2), so a
// stage is 32 KB per CTA instead of 48 KB: a third less operand traffic from L2 and into
// shared memory (96 bytes a cycle of operand reads and 62 of TMA writes against the 128
// that it takes, at the full MMA rate), and six stages instead of four. 75 years, D =
// 3,726, L = 5, k = 20: 6,016 -> 4,949 us; 30 years 1,147 -> 997. The first CTA hands out
// the units and issues the MMAs for both; every role's waits, its own CTA's and the
// other's, are bounded as in a single CTA.
template <int G, bool kWin, bool kBand, bool kLarge, bool kPair>
__global__ void __launch_bounds__(kThreadsG(G), 1)
    fused_tc_kernel(const __grid_constant__ CUtensorMap tmA_hi,
                    const __grid_constant__ CUtensorMap tmA_lo,
                    const __grid_constant__ CUtensorMap tmB_hi,
                    const __grid_constant__ CUtensorMap tmB_lo,
                    const __grid_constant__ TcParams p) {
  extern __shared__ unsigned char smem_raw[];
  const TcArgs& a = p.a;
  const TcWork& w = p.w;
  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  const int NS = p.nstages;
  const int rank = kPair ? (int)ptx::cluster_rank() : 0;

  // ---- shared memory carve-up (ring base aligned to 1 KB for the swizzle pattern)
  const uint32_t raw = ptx::smem_u32(smem_raw);
  const uint32_t ring = (raw + 1023u) & ~1023u;
  unsigned char* gptr = smem_raw + (ring - raw) + (size_t)NS * p.stage_bytes;
  // epilogue regions (one per group), sized for the largest L and k of the call
  const size_t gbytes = group_bytes(a.Lmax);
  uint64_t* bars = reinterpret_cast<uint64_t*>(gptr + G * gbytes);
  const uint32_t full0 = ptx::smem_u32(bars);
  const uint32_t empty0 = full0 + 8u * NS;
  const uint32_t tfull0 = empty0 + 8u * NS;
  const uint32_t tempty0 = tfull0 + 16u;
  const uint32_t drain = tempty0 + 16u;
  const uint32_t qfull0 = drain + 8u;
  const uint32_t qempty0 = qfull0 + 8u * kQueue;
  const uint32_t xfull = qempty0 + 8u * kQueue;  // second group's minima are in (band)
  const uint32_t xempty = xfull + 8u;            // ... and have been read
  const uint32_t pdone = xempty + 8u;            // the pair's second producer has ended
  // units handed out, read by the MMA issuer and the epilogue (16-byte aligned; a
  // negative strip ends the list)
  WorkUnit* qunit = reinterpret_cast<WorkUnit*>(
      (reinterpret_cast<uintptr_t>(bars + 2 * NS + 8 + 2 * kQueue) + 15) & ~uintptr_t(15));
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(qunit + kQueue);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  // the stages the pair's second CTA issued copies for, and their parities
  volatile uint32_t* second = tmem_slot + 2;

  Ctl ctl;
  ctl.abort = abort_flag;
  ctl.err = a.err;
  ctl.limit_ns = (unsigned long long)a.wait_limit_ns;
  ctl.peer_abort = kPair ? ptx::mapa(ptx::smem_u32(tmem_slot + 1), rank ^ 1) : 0u;

  if (threadIdx.x == 0) {
    for (int i = 0; i < NS; ++i) {
      ptx::mbar_init(full0 + 8u * i, 1);
      ptx::mbar_init(empty0 + 8u * i, 1);
    }
    for (int b = 0; b < 2; ++b) {
      ptx::mbar_init(tfull0 + 8u * b, 1);
      // every epilogue thread; in a pair one lane of each of the eight warps
      ptx::mbar_init(tempty0 + 8u * b, kPair ? 8 : kEpiThreads * G);
    }
    ptx::mbar_init(drain, 1);
    for (int i = 0; i < kQueue; ++i) {
      ptx::mbar_init(qfull0 + 8u * i, 1);
      // the MMA thread and each group's leader; in a pair also the second CTA's producer
      ptx::mbar_init(qempty0 + 8u * i, kPair ? 4 : 1 + G);
    }
    ptx::mbar_init(xfull, kEpiThreads);
    ptx::mbar_init(xempty, kEpiThreads);
    ptx::mbar_init(pdone, 1);
    *abort_flag = 0;
    ptx::fence_mbar_init();
    ptx::fence_proxy_async();
  }
  if (warp == 1) {
    if (kPair) {
      ptx::tmem_alloc_pair(ptx::smem_u32(tmem_slot), 512);
      ptx::tmem_relinquish_pair();
    } else {
      ptx::tmem_alloc(ptx::smem_u32(tmem_slot), 512);
      ptx::tmem_relinquish();
    }
    ptx::tc_fence_before();
  }
  if (kPair) ptx::cluster_sync();  // the other CTA's barriers are initialised
  __syncthreads();
  ptx::tc_fence_after();
  launch_wait();  // barriers and tensor memory were set up beside the kernel before
  launch_next();
  const uint32_t tmem_base = *tmem_slot;
  const int nkb = a.Dp / KC;
  const int seg_kb = p.seg_kb;                    // K blocks per accumulation segment
  const int nseg = (nkb + seg_kb - 1) / seg_kb;  // segments per tile
  auto read_unit = [&](int slot) {  // a queue slot, by 16-byte reads
    union {
      int4 v[2];
      WorkUnit u;
    } x;
    x.v[0] = reinterpret_cast<const int4*>(qunit + slot)[0];
    x.v[1] = reinterpret_cast<const int4*>(qunit + slot)[1];
    return x.u;
  };

  if (warp == 0) {
    // ------------------------------------------------------------ producer
    // Hands out units in list order (global counter) through a small queue, so the
    // units in flight across the GPU stay a contiguous window of the list. The whole warp
    // walks the units and waits; an elected lane issues the copies (see the MMA issuer).
    if (ptx::elect_one()) {
      ptx::prefetch_tensormap(&tmA_hi);
      if (!kPair) ptx::prefetch_tensormap(&tmB_hi);
      if (p.split) {
        ptx::prefetch_tensormap(&tmA_lo);
        if (!kPair) ptx::prefetch_tensormap(&tmB_lo);
      }
    }
    const uint64_t pol_a = ptx::l2_policy_evict_last();
    int stage = 0, qs = 0;
    uint32_t phase = 0, qphase = 0, issued = 0, issued_par = 0;
    bool ok = true, withheld = false, first_unit = false;
    UnitSpan us;
    while (ok) {
      if (rank == 0) {
        ok = __all_sync(0xffffffffu, wait_bounded(qempty0 + 8u * qs, qphase ^ 1u, ctl));
        if (!ok) break;
        if (lane == 0) {
          const int u = atomicAdd(w.counter, 1);
          WorkUnit wu;
          if (u < w.nunits) wu = w.units[u];
          else wu.strip = -1;
          if (u == 0) first_unit = true;
          qunit[qs] = wu;
          if (kPair) {
            const uint32_t at = ptx::mapa(ptx::smem_u32(qunit + qs), 1);
            const int4* v = reinterpret_cast<const int4*>(qunit + qs);
            ptx::st_remote(at, v[0]);
            ptx::st_remote(at + 16u, v[1]);
            ptx::mbar_arrive_remote(ptx::mapa(qfull0 + 8u * qs, 1));
          }
          ptx::mbar_arrive(qfull0 + 8u * qs);
        }
        first_unit = __shfl_sync(0xffffffffu, first_unit, 0);
        __syncwarp();
      } else {
        ok = __all_sync(0xffffffffu, wait_bounded<kPair>(qfull0 + 8u * qs, qphase, ctl));
        if (!ok) break;
      }
      const WorkUnit wu = read_unit(qs);
      __syncwarp();
      if (rank && lane == 0) ptx::mbar_arrive_remote(ptx::mapa(qempty0 + 8u * qs, 0));
      if (++qs == kQueue) {
        qs = 0;
        qphase ^= 1u;
      }
      if (wu.strip < 0) break;
      if (!unit_span(wu, p.sr.s, 0, us, rank, w.sym)) continue;
      const int ntiles = us.ntiles, a0 = us.row_base + us.T0;
      for (int it = 0; ok && it < ntiles; ++it) {
        const int c0 = us.row_base + us.jt0 + it * us.adv + (kPair ? rank * BM : 0);
        for (int kb = 0; kb < nkb; ++kb) {
          ok = __all_sync(0xffffffffu, wait_bounded(empty0 + 8u * stage, phase ^ 1u, ctl));
          if (!ok) break;
          if (a.debug_withhold && first_unit && !withheld) {
            withheld = true;  // test hook: unit 0's first stage is never filled
          } else {
            const uint32_t fb = full0 + 8u * stage;
            const uint32_t sb = ring + (uint32_t)stage * p.stage_bytes;
            if (ptx::elect_one()) {
              if (kPair) {
                // both CTAs' copies complete on the first one's barrier
                const uint32_t lb = ptx::mapa(fb, 0);
                if (rank == 0) ptx::mbar_arrive_expect_tx(fb, 2 * p.stage_bytes);
                const uint32_t sB = sb + (p.split ? 2 * kTileA : kTileA);
                ptx::tma_load_2d_pair(sb, &tmA_hi, lb, kb * KC, a0);
                ptx::tma_load_2d_pair(sB, &tmA_hi, lb, kb * KC, c0);
                if (p.split) {
                  ptx::tma_load_2d_pair(sb + kTileA, &tmA_lo, lb, kb * KC, a0);
                  ptx::tma_load_2d_pair(sB + kTileA, &tmA_lo, lb, kb * KC, c0);
                }
              } else {
                ptx::mbar_arrive_expect_tx(fb, p.stage_bytes);
                // the strip operand (A) is read again for every tile of the unit: keep it
                // in L2 ahead of the column tiles when asked to
                if (a.l2_keep_a) {
                  ptx::tma_load_2d_hint(sb, &tmA_hi, fb, kb * KC, a0, pol_a);
                  if (p.split)
                    ptx::tma_load_2d_hint(sb + kTileA, &tmA_lo, fb, kb * KC, a0, pol_a);
                } else {
                  ptx::tma_load_2d(sb, &tmA_hi, fb, kb * KC, a0);
                  if (p.split) ptx::tma_load_2d(sb + kTileA, &tmA_lo, fb, kb * KC, a0);
                }
                if (p.split) {
                  ptx::tma_load_2d(sb + 2 * kTileA, &tmB_hi, fb, kb * KC, c0);
                  ptx::tma_load_2d(sb + 2 * kTileA + kTileB, &tmB_lo, fb, kb * KC, c0);
                } else {
                  ptx::tma_load_2d(sb + kTileA, &tmB_hi, fb, kb * KC, c0);
                }
              }
            }
            issued |= 1u << stage;
            issued_par = (issued_par & ~(1u << stage)) | (phase << stage);
          }
          if (++stage == NS) {
            stage = 0;
            phase ^= 1u;
          }
        }
      }
    }
    // Every copy issued into shared memory must land before a CTA exits. A pair's copies all
    // complete on the first CTA's barriers, so that one waits for both, and neither leaves
    // before (cluster barrier at the end). Where a wait runs out the two producers may have
    // stopped one use of a stage apart: the second says what it issued, and the first, once
    // the abort flag says that nobody relies on the stage, takes the bytes that will never
    // come out of a phase that it armed alone, and arms one for the copies of the second
    // alone. (Neither is ever further ahead: a stage is filled again only once its last
    // contents, of both, were multiplied.)
    if (kPair && rank) {
      __syncwarp();
      if (lane == 0) {
        const uint32_t at = ptx::mapa(ptx::smem_u32(tmem_slot + 2), 0);
        ptx::st_remote_u32(at, issued);
        ptx::st_remote_u32(at + 4u, issued_par);
        ptx::mbar_arrive_remote(ptx::mapa(pdone, 0));
      }
    } else {
      uint32_t i2 = issued, p2 = issued_par;
      if (kPair) {
        if (wait_bounded<true>(pdone, 0, ctl, false)) {
          i2 = second[0];
          p2 = second[1];
        }
        __syncwarp();
      }
      for (int i = 0; i < NS; ++i) {
        const uint32_t fb = full0 + 8u * i;
        const bool own = (issued >> i) & 1u, other = (i2 >> i) & 1u;
        uint32_t par = (issued_par >> i) & 1u;
        if (!own && !other) continue;
        if (kPair && (own != other || ((p2 >> i) & 1u) != par)) {
          const uint64_t t0 = ptx::globaltimer();
          while (!*ctl.abort)
            if (ptx::globaltimer() - t0 > ctl.limit_ns) give_up(ctl);
          __syncwarp();
          // the phase this CTA armed is over: the other one's copies are of the next
          const bool behind =
              __any_sync(0xffffffffu, !own || (other && ptx::mbar_try_wait(fb, par)));
          if (behind) par = (p2 >> i) & 1u;
          if (lane == 0) {
            if (behind) ptx::mbar_arrive_expect_tx(fb, p.stage_bytes);
            else ptx::mbar_complete_tx(fb, p.stage_bytes);
          }
          __syncwarp();
        }
        wait_bounded(fb, par, ctl, false);
      }
    }
    __syncwarp();
  } else if (warp == 1) {
    // ------------------------------------------------------------ MMA issuer
    // The whole warp walks the units and waits; an elected lane issues. Everything an MMA
    // needs is then uniform over the warp, and the instruction takes its descriptors from
    // uniform registers directly: issued by a lane of a divergent branch, each MMA waited
    // for its operands to be moved there and took 172 cycles instead of 128, whatever the
    // data, the clock or the operand traffic.
    if (rank == 0) {
      int stage = 0, qs = 0, gt = 0, acc = 0;
      uint32_t used = 0;  // bit b: parity of the segments that accumulator b has taken
      uint32_t phase = 0, qphase = 0;
      bool ok = true, issued_any = false;
      long long wait_tmem = 0, wait_full = 0;
      const long long t_start = clock64();
      UnitSpan us;
      auto commit = [&](uint32_t b) {
        if (kPair) ptx::mma_commit_pair(b);
        else ptx::mma_commit(b);
      };
      auto mma = [&](uint32_t d, uint64_t da, uint64_t db, uint32_t accumulate) {
        if (kPair) ptx::mma_f16_pair(d, da, db, kIdescPair, accumulate);
        else ptx::mma_f16(d, da, db, kIdesc, accumulate);
      };
      // descriptors of stage 0's operands (a stage or 16 K entries further: a plain offset)
      const uint64_t desc_a = ptx::sdesc_kmajor_sw64(ring);
      const uint64_t desc_b = ptx::sdesc_kmajor_sw64(ring + (p.split ? 2 * kTileA : kTileA));
      constexpr uint32_t kLoA = kTileA >> 4;                         // hi to lo copy
      constexpr uint32_t kLoB = (kPair ? kTileA : kTileB) >> 4;      // (a pair: 128 rows each)
      while (ok) {
        ok = __all_sync(0xffffffffu, wait_bounded(qfull0 + 8u * qs, qphase, ctl));
        if (!ok) break;
        const WorkUnit wu = read_unit(qs);
        __syncwarp();
        if (lane == 0) ptx::mbar_arrive(qempty0 + 8u * qs);
        if (++qs == kQueue) {
          qs = 0;
          qphase ^= 1u;
        }
        if (wu.strip < 0) break;
        if (!unit_span(wu, p.sr.s, 0, us, 0, w.sym)) continue;
        const int ntiles = us.ntiles;
        for (int it = 0; ok && it < ntiles; ++it, ++gt) {
          for (int kb = 0; kb < nkb; ++kb) {
            if (kb % seg_kb == 0) {
              // a new segment: the first of a tile to accumulator gt & 1, others to the other
              if (kb > 0 && ptx::elect_one()) commit(tfull0 + 8u * acc);  // the finished one
              acc = (gt & 1) ^ (kb > 0 ? 1 : 0);
              const long long tw0 = w.stats ? clock64() : 0;
              ok = __all_sync(0xffffffffu, wait_bounded<kPair>(tempty0 + 8u * acc,
                                                               ((used >> acc) & 1u) ^ 1u, ctl));
              used ^= 1u << acc;
              if (!ok) break;
              if (w.stats) wait_tmem += clock64() - tw0;
              ptx::tc_fence_after();
            }
            const uint32_t d = tmem_base + (uint32_t)(acc * BN);
            const long long tf0 = w.stats ? clock64() : 0;
            ok = __all_sync(0xffffffffu, wait_bounded(full0 + 8u * stage, phase, ctl));
            if (!ok) break;
            if (w.stats) wait_full += clock64() - tf0;
            ptx::tc_fence_after();
            const uint32_t off = ((uint32_t)stage * p.stage_bytes) >> 4;
            const uint32_t first = kb % seg_kb == 0 ? 1u : 0u;
            if (ptx::elect_one()) {
#pragma unroll
              for (int kk = 0; kk < KC / 16; ++kk) {
                const uint64_t dah = desc_a + (off + 2 * kk), dbh = desc_b + (off + 2 * kk);
                mma(d, dah, dbh, (first && kk == 0) ? 0u : 1u);
                if (p.split) {
                  mma(d, dah, dbh + kLoB, 1u);
                  mma(d, dah + kLoA, dbh, 1u);
                }
              }
              commit(empty0 + 8u * stage);  // frees the stage once these MMAs finish
            }
            issued_any = true;
            if (++stage == NS) {
              stage = 0;
              phase ^= 1u;
            }
          }
          if (!ok) break;
          if (ptx::elect_one()) commit(tfull0 + 8u * acc);  // the tile's last segment
        }
      }
      if (w.stats && lane == 0) {
        atomicAdd(w.stats + kStatMmaWaitTmem, (unsigned long long)wait_tmem);
        atomicAdd(w.stats + kStatMmaWaitFull, (unsigned long long)wait_full);
        atomicAdd(w.stats + kStatMmaCycles, (unsigned long long)(clock64() - t_start));
      }
      if (issued_any) {
        // all MMAs of the elected lane must finish before TMEM is released (the epilogue,
        // which waits for them otherwise, may have given up)
        if (ptx::elect_one()) {
          if (kPair) ptx::mma_commit_pair_own(drain);
          else ptx::mma_commit(drain);
        }
        wait_bounded(drain, 0, ctl, false);
      }
    }
    __syncwarp();
  } else {
    // ------------------------------------------------------------ epilogue
    const int gid = G == 1 ? 0 : (warp - 2) >> 2;  // epilogue group
    const int q = warp & 3;          // TMEM lane quadrant this warp may access
    const int l = q * 32 + lane;     // accumulator row owned by this thread
    const uint32_t lane_addr = (uint32_t)(q * 32) << 16;
    const int et = threadIdx.x - 64 - kEpiThreads * gid;  // 0..127 within the group
    const int bar = 1 + gid;          // the group's named barrier
    constexpr int kSlots = kLarge && !kBand ? 128 : 64;  // shared minima per row (min_slots)
    // the group's chunks of every tile
    const int ch_lo = gid * (BN / 32 / G), ch_hi = ch_lo + BN / 32 / G;
    // the group's shared memory
    float* Gbuf = reinterpret_cast<float*>(gptr + gid * gbytes);
    float* Wsh = Gbuf + BM * chunk_pitch(a.Lmax, kWin);  // window sums of the tile's output columns
    float* Tsh = Wsh + BN;         // row bounds of the tile's output columns (column side)
    float* Csh = Tsh + BN;         // correction values c of the tile's Gram columns
    ColSide cs;
    cs.cnt = reinterpret_cast<int*>(Csh + BN);
    cs.turn = 0;
    // bit x of word ch: the window sum of the chunk's column x is finite (candidate_masks)
    uint32_t* finite = reinterpret_cast<uint32_t*>(cs.cnt + 64);
    if (et < 64) cs.cnt[et] = 0;  // ordered before their use by a tile's barriers
    int qs = 0, gt = 0;
    uint32_t qphase = 0, xphase = 0;
    bool ok = true;
    UnitSpan us;
    // phase timing of the first epilogue thread (diagnostics)
    // (the two-group form keeps no phase timers: its registers are scarcer)
    const bool timed = G == 1 && w.stats != nullptr && et == 0 && gid == 0;
    long long ph[7] = {0, 0, 0, 0, 0, 0, 0};
    // event counts kept per thread, summed once at the end (diagnostics)
    unsigned int cnt[5] = {0, 0, 0, 0, 0};
    const long long e_start = timed ? clock64() : 0;
    long long tp = e_start;
    auto lap = [&](int i) {
      if (timed) {
        const long long now = clock64();
        ph[i] += now - tp;
        tp = now;
      }
    };
    // this thread has read accumulator b out (in a pair the first CTA's barrier counts the
    // warps of both)
    auto release = [&](int b) {
      ptx::tc_fence_before();
      if (kPair) {
        __syncwarp();
        if (lane == 0) ptx::mbar_arrive_remote(ptx::mapa(tempty0 + 8u * b, 0));
      } else {
        ptx::mbar_arrive(tempty0 + 8u * b);
      }
    };
    uint32_t seen = 0;  // bit b: parity of the segments read from accumulator b
    auto wait_acc = [&](int b) {
      const bool r =
          __all_sync(0xffffffffu, wait_bounded(tfull0 + 8u * b, (seen >> b) & 1u, ctl));
      seen ^= 1u << b;
      return r;
    };
    // Waits for tile gt's segments and adds all to the first one's accumulator, each thread
    // its own row (this group's columns). Formerly the totals were a scratch array in L2,
    // updated by FP32 reductions: D = 58,101, N = 27,394, where the power limit sets the
    // clock, 93.9 -> 90.8 ms (86.2 -> 84.1 a call alone).
    auto collect = [&](int total) -> bool {
      if (!wait_acc(total)) return false;
      ptx::tc_fence_after();
      for (int sg = 1; sg < nseg; ++sg) {
        if (!wait_acc(total ^ 1)) return false;
        ptx::tc_fence_after();
        const uint32_t tT = tmem_base + lane_addr + (uint32_t)(total * BN);
        const uint32_t tU = tmem_base + lane_addr + (uint32_t)((total ^ 1) * BN);
#pragma unroll 1
        for (int c = ch_lo; c < ch_hi; ++c) {
          uint32_t t[32], u[32];
          ptx::tmem_ld32_async(tT + c * 32, t);
          ptx::tmem_ld32_async(tU + c * 32, u);
          ptx::tmem_wait();
#pragma unroll
          for (int x = 0; x < 32; ++x)
            t[x] = __float_as_uint(__uint_as_float(t[x]) + __uint_as_float(u[x]));
          ptx::tmem_st32(tT + c * 32, t);
        }
        ptx::tmem_wait_st();
        release(total ^ 1);
      }
      return true;
    };
    // What a pass over a tile needs from global memory (window sums, bounds and
    // correction values of two of its 256 columns; the row's own values), fetched while
    // the pass before it runs.
    struct Head {
      float w[2], t[2], c[2], wt, cr, thr;
    } hd;
    auto fetch_head = [&](const UnitSpan& s, int it) {
      const int c0 = s.jt0 + it * s.adv, t = s.T0 + l, N = s.M + s.L - 1;
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int x = et + kEpiThreads * h, j = c0 - (s.L - 1) + x;
        const bool in = j >= 0 && j < s.M;
        hd.w[h] = in ? a.W[s.out_base + j] : 0.f;
        hd.t[h] = in ? __uint_as_float(__ldcg(w.thr + s.out_base + j)) : 0.f;
        hd.c[h] = c0 + x < N ? a.cval[s.row_base + c0 + x] : 0.f;  // Gram column day c0 + x
      }
      const bool row_ok = l < s.R && t < s.M;
      hd.wt = row_ok ? a.W[s.out_base + t] : 0.f;
      hd.thr = row_ok ? __uint_as_float(__ldcg(w.thr + s.out_base + t)) : 0.f;
      hd.cr = t < N ? a.cval[s.row_base + t] : 0.f;
    };
    while (ok) {
      bool wok = wait_bounded<kPair>(qfull0 + 8u * qs, qphase, ctl);
      WorkUnit wu;
      wu.strip = -1;
      if (wok) wu = read_unit(qs);
      wok = ptx::named_bar_and(bar, kEpiThreads, wok);  // everyone has read the slot
      if (!wok) {
        ok = false;
        break;
      }
      if (et == 0) {
        if (rank) ptx::mbar_arrive_remote(ptx::mapa(qempty0 + 8u * qs, 0));
        else ptx::mbar_arrive(qempty0 + 8u * qs);
      }
      if (++qs == kQueue) {
        qs = 0;
        qphase ^= 1u;
      }
      if (wu.strip < 0) break;
      if (!unit_span(wu, p.sr.s, 0, us, rank, w.sym)) continue;
      fetch_head(us, 0);
      // Series that share this unit's Gram tiles (several trajectory lengths of one
      // record) are served one after another from the same accumulator; their row
      // lists live for one tile (main units are one tile long; band units keep no lists).
      const int nser = us.nser;
      const int ntiles = us.ntiles;
      RowSide rs;  // this thread's row list in this unit
      GroupMin<kBand && kLarge> gm;
      rs.reset();
      gm.reset();
      for (int it = 0; it < ntiles; ++it, ++gt) {
        lap(6);
        const int acc_l = gt & 1;  // the accumulator of the tile's total
        wok = collect(acc_l);
        wok = ptx::named_bar_and(bar, kEpiThreads, wok);  // all four warps agree
        if (!wok) {
          ok = false;
          break;
        }
        lap(0);
        for (int sj = 0; sj < nser; ++sj) {
        const int L = kWin ? us.L : 1;
        const int LDG = chunk_pitch(L, kWin);
        const int t = us.T0 + l;
        const bool row_ok = l < us.R && t < us.M;
        // the operand layout subtracts groups * c_a * c_b from every Gram entry (see the
        // operand preparation); it is added back when a chunk is read, for every
        // accumulator row whose day exists (halo rows feed other rows' windows)
        // (with one product on split operands the correction entries added
        // +groups c_a c_b: subtract it instead)
        const float crow = (a.corr_neg ? -(float)a.groups : (float)a.groups) * hd.cr;
        const float Wt = hd.wt;
        float thr_row = hd.thr;
        const int jsym = us.T0 + us.R;  // column side from here on (sym)
        const long long cbase = w.sym ? us.col_base + w.col_off[us.strip_base + us.strip] : 0;
        if (nser > 1 || it == 0) {
          rs.reset();
          gm.reset();
          if (!kBand)
            rs.rec = a.part +
                     (size_t)(us.part_base + (long long)t * us.slots + us.slot * G + gid) * a.cap;
        }
        const int c0 = us.jt0 + it * us.adv;
        // W and row bounds of this tile's output columns j = c0 - (L-1) + x (the
        // previous pass's readers passed its last barrier)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          Wsh[et + kEpiThreads * h] = hd.w[h];
          Tsh[et + kEpiThreads * h] = hd.t[h];
          Csh[et + kEpiThreads * h] = hd.c[h];
          const uint32_t f = __ballot_sync(0xffffffffu, hd.w[h] < CUDART_INF_F);
          if (lane == 0) finite[(et >> 5) + 4 * h] = f;
        }
        ptx::named_bar_sync(bar, kEpiThreads);  // read by every thread of the group
        const UnitSpan cu = us;  // this pass; `us` moves on to the next one
        if (sj + 1 < nser) {
          unit_span(wu, p.sr.s, sj + 1, us, rank, w.sym);
          fetch_head(us, it);
        } else if (it + 1 < ntiles) {
          if (nser > 1) unit_span(wu, p.sr.s, 0, us, rank, w.sym);  // (a band unit of several tiles)
          fetch_head(us, it + 1);
        }
        lap(1);
        // chunk ch+1 is fetched while chunk ch is scanned; with two epilogue groups (168
        // registers a thread; the other group hides the latency) when it is read
        const uint32_t tlast = tmem_base + lane_addr + (uint32_t)(acc_l * BN);
        constexpr bool kAhead = G == 1;
        uint32_t vr[32];
        if (kAhead) ptx::tmem_ld32_async(tlast + (uint32_t)(ch_lo * 32), vr);
        float* grow = Gbuf + l * LDG;
#pragma unroll 1
        for (int ch = ch_lo; ch < ch_hi; ++ch) {
          const float* csh = Csh + ch * 32;
          // Gram values of the chunk (correction added back): staged in shared memory
          // for the diagonal window sums, or, with L = 1 (no window), kept in registers
          float c[32];
          if (!kAhead) ptx::tmem_ld32_async(tlast + (uint32_t)(ch * 32), vr);
          ptx::tmem_wait();
#pragma unroll
          for (int x = 0; x < 32; ++x) c[x] = fmaf(crow, csh[x], __uint_as_float(vr[x]));
          if (kWin && L > 1) {
            // the diagonal carry: the L-1 Gram columns before the chunk start its
            // windows: the last ones of the group's previous chunk (of the previous tile
            // of this unit at the tile's first chunk), or, for the second group's first
            // chunk, read from the accumulator
            if (G == 2 && gid == 1 && ch == ch_lo) {
              uint32_t pv[16];
              ptx::tmem_ld16_async(tlast + (uint32_t)(ch_lo * 32 - 16), pv);
              ptx::tmem_wait();
#pragma unroll
              for (int x = 0; x < 16; ++x)
                if (x >= 17 - L) grow[x - (17 - L)] = fmaf(crow, csh[x - 16], __uint_as_float(pv[x]));
            } else if (ch > 0 || (it > 0 && cu.carry)) {
              for (int x = 0; x < L - 1; ++x) grow[x] = grow[32 + x];
            }
#pragma unroll
            for (int x = 0; x < 32; ++x) grow[(L - 1) + x] = c[x];
          }
          if (ch + 1 < ch_hi) {
            if (kAhead) ptx::tmem_ld32_async(tlast + (uint32_t)((ch + 1) * 32), vr);
          } else {
            // the first group's next tile starts from this tile's last columns, which the
            // second group reads: kept in vr until the chunk is done
            if (kWin && G == 2 && gid == 0 && L > 1 && cu.carry && it + 1 < ntiles) {
              uint32_t pv[16];
              ptx::tmem_ld16_async(tlast + (uint32_t)(BN - 16), pv);
              ptx::tmem_wait();
#pragma unroll
              for (int x = 0; x < 16; ++x)
                vr[x] = __float_as_uint(fmaf(crow, Csh[BN - 16 + x], __uint_as_float(pv[x])));
            }
            if (sj == nser - 1) {
              // the accumulator has been read out: hand it back to the MMA warp
              release(acc_l);
            }
          }
          lap(2);
          // the window sums read other rows' staged values (nothing to wait for at L = 1)
          if (kWin && L > 1) ptx::named_bar_sync(bar, kEpiThreads);
          lap(3);
          const int j0 = c0 + ch * 32 - (L - 1);
          // column side of this chunk: output columns j >= jsym inside the unit
          // the first L-1 columns of a unit's first chunk have no carried window
          const int xfirst = (ch == 0 && (it == 0 || !cu.carry)) ? L - 1 : 0;
          const uint32_t unitrange = bit_range(xfirst, 32) & bit_range(cu.jlo - j0, cu.jhi - j0);
          const uint32_t colrange =
              w.sym ? bit_range(jsym - j0, 32) & unitrange : 0u;
          uint32_t cand = 0, ccand = 0;
          if (row_ok && Wt < CUDART_INF_F) {
            // output column x of this chunk is j = j0 + x; its window is the diagonal
            // Gbuf[l+m][x+m], m < L (Eq. 2 as W_t + W_j - 2 sum G)
            if (kWin && L > 1) {
              for (int m = 1; m < L; ++m) {
                const float* gm = grow + m * (LDG + 1);
                if (m == 1) {
#pragma unroll
                  for (int x = 0; x < 32; ++x) c[x] = grow[x] + gm[x];
                } else {
#pragma unroll
                  for (int x = 0; x < 32; ++x) c[x] += gm[x];
                }
              }
            }
            distances(c, Wt, Wsh + ch * 32, kBand ? a.band_margin : 0.f);
            const uint32_t valid = unitrange & finite[ch] & ~bit_range(t - cu.e - j0, t + cu.e + 1 - j0);
            if (kBand) {
              gm.scan(c, valid);  // (outside the exclusion zone)
            } else {
              candidate_masks(c, rs.limit(thr_row), Tsh + ch * 32, cand, ccand);
              cand &= valid;
              ccand &= valid & colrange;
            }
          }
          // every window sum of the chunk is done before a row overwrites the first 32
          // entries of its Gram row (the carried columns 32.. stay) by its distances
          if (kWin && L > 1) ptx::named_bar_sync(bar, kEpiThreads);
          if (!kBand) {
            const uint32_t cmask = ccand;
            if (cand | ccand) store_row<!kWin>(grow, c);
            lap(4);
            cnt[0] += __popc(cand);
            cnt[1] += __popc(ccand);
            const bool over = append<kSlots>(rs, cs, cand, ccand, grow, j0, cu.k, t,
                                             cbase + (j0 - jsym), a.shared_min + cu.out_base + t,
                                             a.shared_min + cu.out_base + j0, w, a);
            if (colrange) {  // the same for the whole group
              const int ne = cs.finish<!kWin>(over, colrange, cmask, c, Gbuf, LDG, l, et, bar,
                                              cu.k, cu.T0, cu.strip, cu.out_base, j0,
                                              cbase + (j0 - jsym), w, a);
              cnt[3] += ne > 0;
              cnt[2] += ne > cu.k;
            }
            rs.compress(cu.k, a, w.thr + cu.out_base + t);
          }
          if (kWin && G == 2 && gid == 0 && L > 1 && ch == ch_hi - 1) {
#pragma unroll
            for (int x = 0; x < 16; ++x)
              if (x >= 17 - L) grow[32 + x - (17 - L)] = __uint_as_float(vr[x]);
          }
          cnt[4] += et == 0;
          lap(5);
        }
        const bool last = nser > 1 || it == ntiles - 1;
        // (main pass, two groups: they hold the same rows and take the refreshes in turn)
        const bool turn = kBand || G == 1 || ((it / a.bound_tiles + cu.slot) & 1) == gid;
        if (turn && (last || (!kBand && (it + 1) % a.bound_tiles == 0))) {
          // a bound of the row's k-th distance: from this unit's columns (band), or from
          // those of every unit so far (main pass)
          float bd = CUDART_INF_F;
          if (!kBand) {
            bd = row_bound<kSlots>(cu.k, a.shared_min + cu.out_base + t, a.out_rows, row_ok,
                                   thr_row);
          } else if (G == 2 && nser == 1) {
            // the second group hands its minima to the first (the chunk buffer of the
            // second group, which the band uses only while it sums windows)
            float* xb = reinterpret_cast<float*>(gptr + gbytes);
            if (gid == 1) {
              ptx::named_bar_sync(bar, kEpiThreads);  // the windows of the last chunk are done
#pragma unroll
              for (int x = 0; x < 32; ++x) xb[x * BM + l] = gm.m[x];
              ptx::mbar_arrive(xfull);
              wok = wait_bounded(xempty, xphase, ctl);  // read: the buffer is free again
            } else {
              wok = wait_bounded(xfull, xphase, ctl);
              if (wok) bd = gm.bound(cu.k, xb + l);
              ptx::mbar_arrive(xempty);
            }
            xphase ^= 1u;
            wok = ptx::named_bar_and(bar, kEpiThreads, wok);
            if (!wok) {
              ok = false;
              break;
            }
          } else {
            bd = gm.bound(cu.k);
          }
          if (row_ok && bd < thr_row && tk_in(cu.out_base + t, a.out_rows, a.err))
            publish_bound(w.thr + cu.out_base + t, bd);
        }
        if (!kBand && last && row_ok && cu.jlo < cu.jhi) {
          const long long li = cu.part_base + (long long)t * cu.slots + cu.slot * G + gid;
          if (tk_in(li, w.part_lists, a.err)) a.part_n[li] = rs.n;
        }
        // the next pass rewrites the tile's W, bounds and correction values
        if (sj + 1 < nser) ptx::named_bar_sync(bar, kEpiThreads);
        }  // series sharing the tile
        if (!ok) break;
      }
      if (!ok) break;
    }
    if (w.stats) {
#pragma unroll
      for (int i = 0; i < 5; ++i) {
        unsigned int v = cnt[i];
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (lane == 0 && v) atomicAdd(w.stats + kStatRowInserts + i, (unsigned long long)v);
      }
    }
    if (timed) {
      lap(6);
      for (int i = 0; i < 6; ++i) atomicAdd(w.stats + kStatEpiWaitAcc + i, (unsigned long long)ph[i]);
      atomicAdd(w.stats + kStatEpiCycles, (unsigned long long)(clock64() - e_start));
    }
  }

  __syncthreads();
  if (kPair) ptx::cluster_sync();  // neither CTA leaves while the other may still reach it
  if (warp == 1) {
    ptx::tc_fence_after();
    if (kPair) ptx::tmem_dealloc_pair(tmem_base, 512);
    else ptx::tmem_dealloc(tmem_base, 512);
  }
}

// ------------------------------------------------------------------- host side
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*,
                                  const cuuint64_t*, const cuuint64_t*, const cuuint32_t*,
                                  const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn() {
  static EncodeTiledFn fn = nullptr;
  if (!fn) {
    void* ptr = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &ptr, 12000, cudaEnableDefault,
                                         &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<EncodeTiledFn>(ptr);
  }
  return fn;
}

// Row-major [N][Dp] BF16 operand copy, boxes of 32 elements x box_rows rows.
bool make_map(CUtensorMap* m, const void* base, int N, int Dp, int box_rows) {
  EncodeTiledFn fn = encode_fn();
  if (!fn) return false;
  const cuuint64_t dims[2] = {(cuuint64_t)Dp, (cuuint64_t)N};
  const cuuint64_t strides[1] = {(cuuint64_t)Dp * 2};
  const cuuint32_t box[2] = {(cuuint32_t)KC, (cuuint32_t)box_rows};
  const cuuint32_t estr[2] = {1, 1};
  return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box,
            estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B,
            CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

size_t epilogue_bytes(int k, int L, int G) {
  return G * group_bytes(L) + 8 * (2 * kMaxStages + 8 + 2 * kQueue) + 16 +
         kQueue * sizeof(WorkUnit) + 16;
}

uint32_t stage_bytes(bool split, bool pair) {
  return (split ? 2 : 1) * (kTileA + (pair ? kTileA : kTileB));
}

int pick_stages(bool split, bool pair, int k, int L, int G) {
  const uint32_t stage = stage_bytes(split, pair);
  const size_t avail = kSmemLimit - 1024 - epilogue_bytes(k, L, G);
  int ns = (int)(avail / stage);
  return ns < kMaxStages ? ns : kMaxStages;
}

template <int G, bool kWin, bool kBand, bool kLarge, bool kPair = false>
cudaError_t launch_g(const CUtensorMap& mAh, const CUtensorMap& mAl, const CUtensorMap& mBh,
                     const CUtensorMap& mBl, const TcParams& p, int num_ctas, size_t smem,
                     cudaStream_t st) {
  const auto kernel = fused_tc_kernel<G, kWin, kBand, kLarge, kPair>;
  cudaError_t err =
      cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (err != cudaSuccess) return err;
  return launch_chained_clusters(kernel, kPair ? 2 : 1, kPair ? num_ctas / 2 * 2 : num_ctas,
                                 kThreadsG(G), smem, st, mAh, mAl, mBh, mBl, p);
}

}  // namespace

bool tc_available() { return encode_fn() != nullptr; }

size_t fused_tc_smem_bytes(bool split, bool pair, int kmax, int Lmax, int G) {
  return 1024 + (size_t)pick_stages(split, pair, kmax, Lmax, G) * stage_bytes(split, pair) +
         epilogue_bytes(kmax, Lmax, G);
}

cudaError_t launch_fused_tc(const void* hi, const void* lo, bool split, const TcArgs& a,
                            const TcWork& w, const SeriesTable& sr, int num_ctas, cudaStream_t st) {
  if (a.Dp % KC != 0) return cudaErrorInvalidValue;
  CUtensorMap mAh, mAl, mBh, mBl;
  if (!make_map(&mAh, hi, a.rows, a.Dp, BM) || !make_map(&mBh, hi, a.rows, a.Dp, BN))
    return cudaErrorNotSupported;
  if (split) {
    if (!make_map(&mAl, lo, a.rows, a.Dp, BM) || !make_map(&mBl, lo, a.rows, a.Dp, BN))
      return cudaErrorNotSupported;
  } else {
    mAl = mAh;
    mBl = mBh;
  }
  thread_local TcParams p;  // large (series table): kept off the stack
  p.a = a;
  p.w = w;
  p.sr = sr;
  p.split = split ? 1 : 0;
  const bool pair = a.pair != 0 && w.write_lists;
  p.stage_bytes = stage_bytes(split, pair);
  const int G = a.egroups;
  if (G != 1 && (G != 2 || a.kmax > 32)) return cudaErrorInvalidValue;
  p.nstages = pick_stages(split, pair, a.kmax, a.Lmax, G);
  if (pair && (G != 1 || num_ctas < 2)) return cudaErrorInvalidValue;
  if (p.nstages < 2) return cudaErrorInvalidValue;
  if (a.seg_k < KC || a.seg_k % KC != 0) return cudaErrorInvalidValue;
  p.seg_kb = a.seg_k / KC;
  const size_t smem = fused_tc_smem_bytes(split, pair, a.kmax, a.Lmax, G);
  const bool win = a.Lmax > 1, band = !w.write_lists, large = a.kmax > (band ? 32 : 40);
  auto go = [&](auto fn) { return fn(mAh, mAl, mBh, mBl, p, num_ctas, smem, st); };
  if (G == 2) {
    if (band) return win ? go(launch_g<2, true, true, false>) : go(launch_g<2, false, true, false>);
    return win ? go(launch_g<2, true, false, false>) : go(launch_g<2, false, false, false>);
  }
  if (pair) {
    if (large)
      return win ? go(launch_g<1, true, false, true, true>) : go(launch_g<1, false, false, true, true>);
    return win ? go(launch_g<1, true, false, false, true>) : go(launch_g<1, false, false, false, true>);
  }
  if (large) {
    if (band) return win ? go(launch_g<1, true, true, true>) : go(launch_g<1, false, true, true>);
    return win ? go(launch_g<1, true, false, true>) : go(launch_g<1, false, false, true>);
  }
  if (band) return win ? go(launch_g<1, true, true, false>) : go(launch_g<1, false, true, false>);
  return win ? go(launch_g<1, true, false, false>) : go(launch_g<1, false, false, false>);
}

}  // namespace traknn
