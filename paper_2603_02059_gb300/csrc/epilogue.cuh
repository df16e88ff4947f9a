// epilogue.cuh -- per-row work that turns a tile of the snapshot Gram matrix into
// trajectory distances and keeps each row's candidates for its k nearest: the candidate
// lists of the symmetric kernels (RowSide, ColSide), and the plain per-row scan of the
// FP32 kernel that evaluates both triangles.
//
// With day norms n_a = ||X_a||^2 and window sums W_t = sum_{m<L} n_{t+m}, the
// trajectory distance of Eq. 2 expands (Eq. 4 applied to every day pair) into
//     D(t,j) = W_t + W_j - 2 sum_{m<L} G(t+m, j+m),   G(a,b) = <X_a, X_b>.
// The sum runs down one diagonal of G. It is evaluated explicitly, L terms per
// output, from Gram values held on chip (the current tile plus the last L-1
// columns carried over from the previous tile of the same row strip), so there
// is no running add/subtract chain and no drift however long the diagonal is.
#pragma once

#include <cuda_runtime.h>
#include <math_constants.h>
#include <stdint.h>

#include "internal.h"
#include "tc_ptx.cuh"

namespace traknn {

// A sorted (ascending distance) list of k candidates per owning thread, kept in
// shared memory as [k][stride] so that consecutive threads use consecutive banks.
// Empty slots hold (+inf, -1).
struct SmemList {
  float* d;
  int32_t* i;
  int stride;
  int k;

  __device__ __forceinline__ void reset(int tid) const {
    for (int p = 0; p < k; ++p) {
      d[p * stride + tid] = CUDART_INF_F;
      i[p * stride + tid] = -1;
    }
  }

  __device__ __forceinline__ float threshold(int tid) const { return d[(k - 1) * stride + tid]; }

  // Insert (dv, jv) with dv < threshold. Candidates reach a list in increasing
  // index order, so stopping at an equal distance keeps the smaller index first:
  // the list stays sorted by (distance, index) (Algorithm 1, kNN step).
  // Returns the new threshold (the k-th distance).
  __device__ __forceinline__ float insert(int tid, float dv, int32_t jv) const {
    int p = k - 1;
    while (p > 0) {
      float q = d[(p - 1) * stride + tid];
      if (!(q > dv)) break;
      d[p * stride + tid] = q;
      i[p * stride + tid] = i[(p - 1) * stride + tid];
      --p;
    }
    d[p * stride + tid] = dv;
    i[p * stride + tid] = jv;
    return d[(k - 1) * stride + tid];
  }

  // Insert (dv, jv) in (distance, index) order when candidates arrive in any
  // index order. Requires (dv, jv) to precede the current k-th entry.
  __device__ __forceinline__ float insert_key(int tid, float dv, int32_t jv) const {
    int p = k - 1;
    while (p > 0) {
      const float q = d[(p - 1) * stride + tid];
      const int32_t qi = i[(p - 1) * stride + tid];
      if (!(q > dv || (q == dv && qi > jv))) break;
      d[p * stride + tid] = q;
      i[p * stride + tid] = qi;
      --p;
    }
    d[p * stride + tid] = dv;
    i[p * stride + tid] = jv;
    return d[(k - 1) * stride + tid];
  }
};

struct RowCtx {
  int t;        // output trajectory row
  float Wt;     // window sum of row t
  int lrow;     // row of the G buffer holding day t
  int L, e;
  int jlo, jhi; // output columns owned by the current unit
};

// Output columns x in [x0, x1) of one tile for one row. `g` points at the G
// buffer column that holds Gram column j0 (the output column of x = 0); the
// window for output x reads g[(lrow+m)*ldg + x + m], m < L.
__device__ __forceinline__ void window_topk(const float* g, int ldg, const RowCtx& rc, int x0,
                                            int x1, int j0, const float* __restrict__ W,
                                            const SmemList& list, int tid, float& thr) {
  for (int x = x0; x < x1; ++x) {
    const int j = j0 + x;
    if (j < rc.jlo || j >= rc.jhi) continue;
    const int gap = rc.t > j ? rc.t - j : j - rc.t;
    if (gap <= rc.e) continue;
    const float* gp = g + rc.lrow * ldg + x;
    float c = gp[0];
    for (int m = 1; m < rc.L; ++m) c += gp[m * (ldg + 1)];
    const float dc = fmaf(-2.0f, c, rc.Wt + __ldg(W + j));
    const float dv = dc < 0.0f ? 0.0f : dc;  // (a NaN stays one: below no threshold)
    if (dv < thr) thr = list.insert(tid, dv, j);
  }
}

// -------------------------------------------------------------------- work units
// A unit with its series' parameters.
struct UnitSpan {
  int strip, T0, jt0, jlo, jhi, ntiles, slot, nser, step;  // jt0: first Gram column
  int carry, adv;  // carry: the last L-1 Gram columns pass from tile to tile; adv: tile stride
  int M, L, k, e, R;      // series: trajectories, length, neighbours, exclusion, rows per strip
  int row_base, out_base, slots, strip_base;
  long long part_base, col_base;
};

// Unit wu for the sj-th of the series that share its Gram tiles (sj = 0: the one
// with the most trajectories, whose tiles cover the others').
// A unit of a pair of CTAs covers two strips with the Gram tiles of the first; `rank` 1 is
// the second one, whose own output columns start later (sym).
__device__ __forceinline__ bool unit_span(const WorkUnit& wu, const SeriesInfo* sr, int sj,
                                          UnitSpan& us, int rank = 0, int sym = 0) {
  const SeriesInfo& si = sr[wu.series + sj];
  us.nser = wu.pad[0] > 1 ? wu.pad[0] : 1;
  us.M = si.M;
  us.L = si.L;
  us.k = si.k;
  us.e = si.e;
  us.R = si.rows_out;
  us.row_base = si.row_base;
  us.out_base = si.out_base;
  us.slots = si.slots;
  us.strip_base = si.strip_base;
  us.part_base = si.part_base;
  us.col_base = si.col_base;
  us.strip = wu.strip + rank;
  us.T0 = us.strip * us.R;
  us.jt0 = wu.jlo;
  us.jlo = rank && sym ? max(wu.jlo, us.T0) : wu.jlo;
  us.jhi = min(wu.jhi, si.M);
  us.slot = wu.slot;
  us.step = si.step;
  if (rank && wu.pad[1] == 0) us.R = 0;  // the pair's second strip is not of this launch
  if (us.jt0 >= us.jhi) return false;
  // A unit of one series: Gram tiles follow each other without overlap, tile it
  // covering Gram columns [jlo + 256 it, jlo + 256 (it+1)); the epilogue carries the
  // last L-1 columns of a tile into the next, so the windows of all output columns
  // [jlo, jhi) are complete once Gram column jhi + L - 2 is in. A unit shared by
  // several series (each restages the chunk buffer with its own L) has no carry: its
  // tiles overlap by the largest L - 1 and each yields `step` output columns.
  us.carry = us.nser == 1;
  us.adv = us.carry ? kTileCols : us.step;
  us.ntiles = us.carry ? (us.jhi - us.jt0 + us.L - 1 + kTileCols - 1) / kTileCols
                       : (us.jhi - us.jt0 + us.step - 1) / us.step;
  return true;
}

// ---------------------------------------------------------------- candidate lists
// The symmetric kernels do not sort while they scan. A row appends every distance within
// its current bound to an unsorted list of its own in global memory (one 8-byte store; no
// lane waits for another); bounds come from minima over groups of columns, and a warp cuts a
// list to its smallest entries only when it runs full; the merge kernel selects the exact
// k nearest from all lists. What bounds this part is the instruction count per candidate: at
// 75 years of 32 values, L = 5, k = 20 (about 340 row and 250 column candidates per row) the
// former sorted register list took a 20-step bubble of compares and selects per candidate.

// Bits [lo, hi) of a 32-bit word (empty when hi <= lo).
__device__ __forceinline__ uint32_t bit_range(int lo, int hi) {
  lo = max(lo, 0);
  hi = min(hi, 32);
  if (hi <= lo) return 0u;
  const uint32_t w = (hi - lo >= 32) ? 0xffffffffu : ((1u << (hi - lo)) - 1u);
  return w << lo;
}

// Publish an upper bound of a row's k-th distance. The same pair distance can be
// evaluated more than once (band pre-pass and main pass; a pair and its transpose)
// with results a few ulp apart, so a bound taken from one evaluation is widened by
// a relative 2^-12 (far above those differences) before it prunes another; a wider
// bound only admits more candidates to the exact final selection.
__device__ __forceinline__ void publish_bound(unsigned int* thr, float d) {
  atomicMin(thr, __float_as_uint(__fmul_ru(d, 1.0f + 0x1p-12f)));
}

// Window sums c[x] = C(t, j0 + x) of one row to distances W_t + W_j - 2 C, not yet
// clamped at 0 (a clamped value is a candidate if and only if the unclamped one is: every
// bound is >= 0). With margin > 0 (one-product band pre-pass) the distance raised by a
// bound of its error. w: window sums of the 32 columns, 16-byte aligned.
__device__ __forceinline__ void distances(float (&c)[32], float Wt, const float* w, float margin) {
#pragma unroll
  for (int x4 = 0; x4 < 8; ++x4) {
    const float4 w4 = reinterpret_cast<const float4*>(w)[x4];
    const float wv[4] = {w4.x, w4.y, w4.z, w4.w};
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      const int x = 4 * x4 + u;
      const float s = Wt + wv[u];
      c[x] = fmaf(-2.0f, c[x], s);
      if (margin != 0.f) c[x] = fmaf(margin, s, fmaxf(c[x], 0.0f)) * (1.0f + 0x1p-20f);
    }
  }
}

// Bit x of cand: d[x] <= lim; of ccand: d[x] <= t[x] (t 16-byte aligned). The sign of the
// difference is shifted in with one funnel shift: the difference runs on the FMA pipe,
// where a compare and a select would both take the half-rate ALU pipe. A NaN distance would
// pass (its difference has a clear sign): the caller masks the rows and columns whose window
// sum is not finite, which are those of a NaN distance. (The reversed difference, which
// no NaN passes, took 1.2 % more of a 75-year call of 32 values, a compare per candidate in
// `append` 1.2 % of a BF16 one; one word of finite columns per chunk 0.1 %.)
__device__ __forceinline__ void candidate_masks(const float (&d)[32], float lim, const float* t,
                                                uint32_t& cand, uint32_t& ccand) {
  uint32_t a = 0, b = 0;
#pragma unroll
  for (int x4 = 7; x4 >= 0; --x4) {
    const float4 t4 = reinterpret_cast<const float4*>(t)[x4];
    const float tv[4] = {t4.x, t4.y, t4.z, t4.w};
#pragma unroll
    for (int u = 3; u >= 0; --u) {
      const int x = 4 * x4 + u;
      a = __funnelshift_l(__float_as_uint(lim - d[x]), a, 1);
      b = __funnelshift_l(__float_as_uint(tv[u] - d[x]), b, 1);
    }
  }
  cand = ~a;
  ccand = ~b;
}

// This row's 32 distances to its row of the chunk buffer.
template <bool kVec>
__device__ __forceinline__ void store_row(float* row, const float (&d)[32]) {
  if (kVec) {
#pragma unroll
    for (int x = 0; x < 8; ++x)
      reinterpret_cast<float4*>(row)[x] =
          make_float4(d[4 * x], d[4 * x + 1], d[4 * x + 2], d[4 * x + 3]);
  } else {
#pragma unroll
    for (int x = 0; x < 32; ++x) row[x] = d[x];
  }
}

constexpr int kListRegs = 4;  // entries of one list per lane (list_cap is at most 128)

__device__ __forceinline__ void list_load(const int2* rec, int n, unsigned (&db)[kListRegs],
                                          int (&ix)[kListRegs]) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int u = 0; u < kListRegs; ++u) {
    const int q = lane + 32 * u;
    db[u] = 0xFFFFFFFFu;
    ix[u] = 0;
    if (q < n) {
      const int2 e = __ldcg(rec + q);
      ix[u] = e.x;
      db[u] = (unsigned)e.y & 0x7FFFFFFFu;
    }
  }
}

// By a whole warp: the bits T of a distance such that between k and most of the loaded
// entries (n >= k of them) are at or below it, or, where ties leave no such distance, of
// the k-th smallest one. Distances are >= 0, so their bit patterns order like the values.
__device__ __forceinline__ unsigned list_bound(const unsigned (&db)[kListRegs], int k, int most) {
  unsigned lo = 0xFFFFFFFFu, hi = 0;
#pragma unroll
  for (int u = 0; u < kListRegs; ++u) {
    lo = min(lo, db[u]);
    hi = max(hi, db[u] == 0xFFFFFFFFu ? 0u : db[u]);
  }
  lo = __reduce_min_sync(0xffffffffu, lo);
  hi = __reduce_max_sync(0xffffffffu, hi);
  // Three thresholds a step: their counts (at most 128 each) share a word, and so one
  // reduction, whose latency is most of a step (against one threshold: four lengths at 30
  // years 1,661 -> 1,641 us, 20 years BF16 544 -> 539, five years of 16 x 32 122.3 -> 121.0).
  while (lo < hi) {
    const unsigned d = hi - lo, m1 = lo + (d >> 2), m2 = lo + (d >> 1), m3 = m2 + (d >> 2);
    unsigned n = 0;
#pragma unroll
    for (int u = 0; u < kListRegs; ++u)
      n += (db[u] <= m1 ? 1u : 0u) + (db[u] <= m2 ? 1u << 8 : 0u) + (db[u] <= m3 ? 1u << 16 : 0u);
    n = __reduce_add_sync(0xffffffffu, n);
    const int c1 = n & 0xFF, c2 = (n >> 8) & 0xFF, c3 = n >> 16;
    if (c3 < k) {
      lo = m3 + 1;
      continue;
    }
    const int c = c1 >= k ? c1 : c2 >= k ? c2 : c3;
    if (c1 < k) lo = (c2 >= k ? m1 : m2) + 1;
    hi = c1 >= k ? m1 : c2 >= k ? m2 : m3;
    if (c <= most) break;
  }
  return hi;
}

// One thread's row list in the current work unit. Every lane of a warp calls each
// function; lanes without a row keep n = 0.
struct RowSide {
  int2* rec;    // the list (a.cap entries)
  int n;        // entries
  float bound;  // at least k entries of the list are at or below it (+inf: none known)

  __device__ __forceinline__ void reset() {
    n = 0;
    bound = CUDART_INF_F;
  }
  // A distance enters the list if it is <= limit: below `bound` (an equal distance of a
  // larger index cannot be among the k nearest) and within the row's published bound.
  __device__ __forceinline__ float limit(float thr_row) const {
    const float below = bound > 0.f ? __uint_as_float(__float_as_uint(bound) - 1u) : -CUDART_INF_F;
    return fminf(below, thr_row);
  }
  // Cuts the lists of this warp that have no room for another chunk.
  __device__ __forceinline__ void compress(int k, const TcArgs& a, unsigned int* thr) {
    const int room = a.cap - 32;
    unsigned full = __ballot_sync(0xffffffffu, n > room);
    if (!full) return;  // the usual case
    const int lane = threadIdx.x & 31;
    __syncwarp();
    while (full) {
      const int src = __ffs(full) - 1;
      full &= full - 1;
      int2* r = reinterpret_cast<int2*>(
          __shfl_sync(0xffffffffu, reinterpret_cast<unsigned long long>(rec), src));
      const int m = __shfl_sync(0xffffffffu, n, src);
      unsigned db[kListRegs];
      int ix[kListRegs];
      list_load(r, m, db, ix);
      const unsigned T = list_bound(db, k, room);
      // kept: everything below T and, if those at T make it too many (ties), only the
      // first of them (the smallest indices) up to k entries
      int lt = 0, le = 0;
#pragma unroll
      for (int u = 0; u < kListRegs; ++u) {
        lt += db[u] < T ? 1 : 0;
        le += db[u] <= T ? 1 : 0;
      }
      lt = __reduce_add_sync(0xffffffffu, lt);
      le = __reduce_add_sync(0xffffffffu, le);
      int ties = le > room ? k - lt : le;  // entries equal to T that may stay
      int base = 0;
#pragma unroll
      for (int u = 0; u < kListRegs; ++u) {
        const unsigned below = (1u << lane) - 1u;
        const unsigned eq = __ballot_sync(0xffffffffu, db[u] == T);
        const bool keep = db[u] < T || (db[u] == T && __popc(eq & below) < ties);
        ties -= __popc(eq);
        const unsigned kb = __ballot_sync(0xffffffffu, keep);
        if (keep) r[base + __popc(kb & below)] = make_int2(ix[u], (int)db[u]);
        base += __popc(kb);
      }
      if (lane == src) {
        n = base;
        bound = __uint_as_float(T);
        publish_bound(thr, bound);
      }
    }
    __syncwarp();
  }
};

// An upper bound of the k-th smallest of the values `each` hands to its argument: the k-th
// smallest, or up to 2^-10 of their spread above it. Values from 3e38 on (the fill
// pattern of unused slots, +inf) do not count; +inf if there are fewer than k others.
template <class Each>
__device__ __forceinline__ float kth_bound(int k, Each&& each) {
  float lo = CUDART_INF_F, hi = -CUDART_INF_F;
  int n = 0;
  each([&](float v) {
    lo = fminf(lo, v);
    hi = fmaxf(hi, v < 3e38f ? v : -CUDART_INF_F);
    n += v < 3e38f ? 1 : 0;
  });
  if (n < k) return CUDART_INF_F;
#pragma unroll 1
  for (int step = 0; step < 10; ++step) {
    const float mid = 0.5f * lo + 0.5f * hi;
    int c = 0;
    each([&](float v) { c += v <= mid ? 1 : 0; });
    if (c >= k) hi = mid;
    else lo = mid;
  }
  return fmaxf(hi, 0.f);
}

// Bounds without lists (band pre-pass). A row's scanned columns fall into 32 groups (the column's place in
// its chunk of 32); the thread keeps each group's smallest distance in a register, so k of
// these minima are k distances of different columns and the k-th smallest minimum bounds
// the row's k-th distance: one minimum per distance, no branch and no memory access, where
// a sorted list costs a bubble per candidate. For k = 20 the bound of 32 groups of 64
// columns is on average that of the 31st nearest column instead of the 20th. kTop2 (k > 32)
// keeps each group's two smallest.
template <bool kTop2>
struct GroupMin {
  float m[32];
  float m2[kTop2 ? 32 : 1];

  __device__ __forceinline__ void reset() {
#pragma unroll
    for (int x = 0; x < 32; ++x) m[x] = CUDART_INF_F;
#pragma unroll
    for (int x = 0; x < (kTop2 ? 32 : 1); ++x) m2[x] = CUDART_INF_F;
  }
  __device__ __forceinline__ void add(int x, float d) {
    if (kTop2) m2[x] = fminf(m2[x], fmaxf(m[x], d));
    m[x] = fminf(m[x], d);
  }
  // The distances of one chunk whose bit in `valid` is set.
  __device__ __forceinline__ void scan(const float (&d)[32], uint32_t valid) {
    if (valid == 0xFFFFFFFFu) {
#pragma unroll
      for (int x = 0; x < 32; ++x) add(x, d[x]);
    } else if (valid) {
#pragma unroll
      for (int x = 0; x < 32; ++x) add(x, (valid >> x) & 1u ? d[x] : CUDART_INF_F);
    }
  }
  // An upper bound of the k-th smallest distance scanned (+inf: fewer than k minima). With
  // `other`, 32 more minima of other columns of the same row ([32][128], this row's column).
  __device__ __forceinline__ float bound(int k, const float* other = nullptr) const {
    float o[32];
    if (other) {
#pragma unroll
      for (int x = 0; x < 32; ++x) o[x] = other[x * 128];
    }
    return kth_bound(k, [&](auto&& f) {
#pragma unroll
      for (int x = 0; x < 32; ++x) f(m[x]);
      if (kTop2) {
#pragma unroll
        for (int x = 0; x < (kTop2 ? 32 : 1); ++x) f(m2[x]);
      }
      if (other) {
#pragma unroll
        for (int x = 0; x < 32; ++x) f(o[x]);
      }
    });
  }
};

// Main pass: the bounds of all units of a row together. Every candidate, row or column
// side, also lowers one of its row's `slots` shared minima, shared_min[slot][row] (a
// distance above the row's bound could not lower it). Every pair is evaluated once in the
// main pass, so no column counts twice whatever slot it takes; the k-th smallest slot
// bounds the row's k-th distance over everything evaluated so far, by any unit, so units
// running side by side profit from one another: with the bounds of a 512-column band alone
// a warp's 32 x 32 outputs hold about 27 row candidates (75 years, D = 3,726, k = 20), with
// those of half of all columns 1.4.
//
// row_bound: that bound for one row per thread (by whole warps; `min` points at the row),
// if it is at least 3 % below `thr`, else `thr`. A first count decides whether any row of
// the warp can gain; the search then stops at thr / 64.
template <int S>
__device__ __forceinline__ float row_bound(int k, const unsigned* min, long long stride, bool row,
                                           float thr) {
  float o[S];
#pragma unroll
  for (int x = 0; x < S; ++x)
    o[x] = row ? __uint_as_float(__ldcg(min + x * stride)) : CUDART_INF_F;
  if (__any_sync(0xffffffffu, row && thr > 3e38f)) {  // rows without a bound yet
    const float b = kth_bound(k, [&](auto&& f) {
#pragma unroll
      for (int x = 0; x < S; ++x) f(o[x]);
    });
    return fminf(thr, b);
  }
  auto count = [&](float mid) {
    int c = 0;
#pragma unroll
    for (int x = 0; x < S; ++x) c += o[x] <= mid ? 1 : 0;
    return c;
  };
  float hi = thr, lo = 0.5f * thr, mid = 0.97f * thr;
#pragma unroll 1
  for (int step = 0; step < 6; ++step) {
    const bool in = count(mid) >= k;
    if (step == 0 && !__any_sync(0xffffffffu, in)) return thr;
    if (in) hi = mid;
    else lo = mid;
    mid = 0.5f * lo + 0.5f * hi;
  }
  return hi;
}

// Column-side lists of one epilogue group (128 threads): the columns of a chunk, beyond
// the strip's own block, take the rows within their bound. A chunk holds all 128 rows of
// its 32 columns, so a column's list (one record of col_pitch ints) is complete when the
// chunk is: a row takes its place in it from a shared-memory counter. More than k
// candidates (rare once bounds are known) are cut to the k best by a warp. Each candidate
// also lowers the column's shared minima (row_bound).
struct ColSide {
  int* cnt;      // [2][32] counters: one set per chunk, taken in turn
  int turn;

  __device__ __forceinline__ int* counters() const { return cnt + 32 * (turn & 1); }

  // Ends a chunk (called by the whole group): counts, masks and bounds of its columns
  // (colrange), the k best of the overfull ones. cmask and dist: this row's column-side
  // candidates and distances; buf: the chunk buffer, this thread's row l. Returns the
  // number of candidates of this thread's column (0: none or no column).
  template <bool kVec>
  __device__ __forceinline__ int finish(bool over, uint32_t colrange, uint32_t cmask,
                                        float (&dist)[32], float* buf, int pitch, int l, int et,
                                        int bar, int k, int T0, int strip, int out_base, int j0,
                                        long long first, const TcWork& w, const TcArgs& a) {
    const int lane = threadIdx.x & 31;
    const int x = (et >> 5) * 8 + (lane & 7);  // column of lanes 0..7
    const bool own = lane < 8 && ((colrange >> x) & 1u);
    const long long rec = (first + x) * col_pitch(w.kstride);
    unsigned int* thr = w.thr + out_base + j0 + x;
    int* c = counters();
    ++turn;
    if (ptx::named_bar_or(bar, 128, over)) {
#pragma unroll
      for (int y = 0; y < 32; ++y) dist[y] = (cmask >> y) & 1u ? fmaxf(dist[y], 0.0f) : CUDART_INF_F;
      store_row<kVec>(buf + l * pitch, dist);
      ptx::named_bar_sync(bar, 128);
      // the overfull columns, shared out among the four warps: the column's 128 distances,
      // four per lane in row order, cut to the k smallest (the first ones among ties)
      unsigned todo = __ballot_sync(0xffffffffu, c[lane] > k) & (0x11111111u << (et >> 5));
      while (todo) {
        const int y = __ffs(todo) - 1;
        todo &= todo - 1;
        unsigned db[kListRegs];
        int lt = 0;
#pragma unroll
        for (int u = 0; u < kListRegs; ++u) {
          const float v = buf[(lane + 32 * u) * pitch + y];
          db[u] = v < CUDART_INF_F ? __float_as_uint(v) & 0x7FFFFFFFu : 0xFFFFFFFFu;
        }
        const unsigned T = list_bound(db, k, k);
#pragma unroll
        for (int u = 0; u < kListRegs; ++u) lt += db[u] < T ? 1 : 0;
        int ties = k - __reduce_add_sync(0xffffffffu, lt), base = 0;
        const long long at = (first + y) * col_pitch(w.kstride) + 2;
#pragma unroll
        for (int u = 0; u < kListRegs; ++u) {
          const unsigned below = (1u << lane) - 1u;
          const unsigned eq = __ballot_sync(0xffffffffu, db[u] == T);
          const bool keep = db[u] < T || (db[u] == T && __popc(eq & below) < ties);
          ties -= __popc(eq);
          const unsigned kb = __ballot_sync(0xffffffffu, keep);
          const int pos = base + __popc(kb & below);
          if (keep && tk_in(at + 2 * pos + 1, w.col_ints, a.err))
            *reinterpret_cast<int2*>(w.col_rec + at + 2 * pos) =
                make_int2(T0 + lane + 32 * u, (int)db[u]);
          base += __popc(kb);
        }
        if (lane == 0 && tk_in(out_base + j0 + y, a.out_rows, a.err))
          publish_bound(w.thr + out_base + j0 + y, __uint_as_float(T));
      }
      ptx::named_bar_sync(bar, 128);  // the rows are read no more
    }
    if (!own) return 0;
    const int ne = c[x];
    if (ne == 0) return 0;  // an empty list gets no record: its mask bit stays clear
    c[x] = 0;
    if (tk_in(rec, w.col_ints, a.err)) w.col_rec[rec] = min(ne, k);
    const long long mi = (long long)(out_base + j0 + x) * w.mask_words + (strip >> 5);
    if (tk_in(mi, (long long)a.out_rows * w.mask_words, a.err))
      atomicOr(w.col_mask + mi, 1u << (strip & 31));
    if (ne == k) {  // exactly k candidates: the largest bounds the column's k-th distance
      float mx = 0.f;
      for (int p = 0; p < k; ++p)
        if (tk_in(rec + 3 + 2 * p, w.col_ints, a.err))
          mx = fmaxf(mx, __int_as_float(__ldcg(w.col_rec + rec + 3 + 2 * p)));
      if (tk_in(out_base + j0 + x, a.out_rows, a.err)) publish_bound(thr, mx);
    }
    return ne;
  }
};

// This row's candidates of one chunk (bits of cand: for the row's list; of ccand: for the
// columns' lists) into the lists and the shared minima, S slots a row. One loop takes both
// sides: a distance that is close for its row is often close for its column too. drow: the
// row's distances; t: the row; first: the column list of the chunk's column 0 (output column
// j0); rmin, cmin: the shared minima of the row and of column j0. Returns whether a column
// is overfull.
//
// The warp runs as many rounds as its fullest row has candidates (two or three), without
// divergent branches: a round's latency is what the loop costs, so the next distance is
// read a round ahead and the column's counter is asked before the row's stores.
template <int S>
__device__ __forceinline__ bool append(RowSide& rs, const ColSide& cs, uint32_t cand,
                                       uint32_t ccand, const float* drow, int j0, int k, int t,
                                       long long first, unsigned* rmin, unsigned* cmin,
                                       const TcWork& w, const TcArgs& a) {
  uint32_t both = cand | ccand;
  const int rounds = __reduce_max_sync(0xffffffffu, __popc(both));
  if (rounds == 0) return false;
  int* c = cs.counters();
  const int cp = col_pitch(w.kstride) / 2;  // in entries
  const long long at0 = first * cp + 1;
  int2* col = reinterpret_cast<int2*>(w.col_rec) + at0;
  unsigned* cm = cmin + (long long)(t & (S - 1)) * a.out_rows;
  bool over = false;
  int x = both ? __ffs(both) - 1 : 0;
  float v = drow[x];
  for (int i = 0; i < rounds; ++i) {
    const bool act = both != 0;
    const bool row = act && ((cand >> x) & 1u), cl = act && ((ccand >> x) & 1u);
    const int y = x, dv = __float_as_int(fmaxf(v, 0.0f));
    const unsigned bits = (unsigned)dv & 0x7FFFFFFFu;
    int pos = 0;
    if (cl) pos = atomicAdd(c + y, 1);
    both &= both - 1u;
    x = both ? __ffs(both) - 1 : 0;
    v = drow[x];
    if (row) {
      atomicMin(rmin + (long long)((j0 + y) & (S - 1)) * a.out_rows, bits);
      if (tk_in(rs.n, a.cap, a.err)) rs.rec[rs.n] = make_int2(j0 + y, dv);
    }
    rs.n += row ? 1 : 0;
    if (cl) atomicMin(cm + y, bits);
    if (cl && pos < k && tk_in(2 * (at0 + y * cp + pos) + 1, w.col_ints, a.err))
      col[y * cp + pos] = make_int2(t, dv);
    over |= cl && pos >= k;
  }
  return over;
}

}  // namespace traknn
