// kernel_fp32.cu -- the plain FP32 path: CUDA-core FMA Gram tiles (Algorithm 1,
// "Symmetric Batched GeMM") fused with the trajectory-distance window, the
// exclusion mask and the candidate lists (Algorithm 1, kNN step). The N x N
// snapshot matrix never leaves the chip.
//
// Two kernels share the Gram code. fused_fp32_kernel walks the work units of the
// tensor-core path (upper triangle only, epilogue.cuh): one persistent CTA per SM computes
// a unit's 128 x 256 Gram tiles in two halves into shared memory, beside the L-1 columns
// carried from the previous tile, and two groups of 128 threads, one thread per row, scan
// 128 columns each. fused_fp32_both_kernel evaluates both triangles in 128 x 128 tiles
// with sorted lists in shared memory: the form of the entry point whose scratch is fixed, and
// of the shortest calls (one tile per CTA and no band before it).
//
// What bounds both is the FP32 FMA rate; a Gram entry's products are summed in the same
// order in either triangle and either kernel, so G(a, b) = G(b, a) bit for bit and the
// symmetric kernel's results equal those of the other.
#include <cuda_runtime.h>
#include <math_constants.h>

#include "epilogue.cuh"
#include "internal.h"

namespace traknn {
namespace {

constexpr int BM = kTileRows;  // Gram rows per tile
constexpr int BN = 128;        // Gram columns per half tile
constexpr int BK = 16;         // depth of one shared-memory stage
constexpr int NT = 256;        // threads
constexpr int LDA = BM + 4;
constexpr int kPitchBoth = kHalo + BN + 1;   // odd row pitches: conflict-free diagonal reads
constexpr int kPitch = kHalo + 2 * BN + 1;
constexpr int kRowPitch = 36;  // a row of 32 distances (16-byte aligned, conflict-free)

struct Stages {
  float As[2][BK][LDA];
  float Bs[2][BK][LDA];
};

__device__ __forceinline__ void load_stage(const float* __restrict__ Xc, int r_end, int c_end,
                                           int Dp, int r0, int c0, int k0, int tid,
                                           float4 (&ra)[2], float4 (&rb)[2]) {
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    const int f = tid + q * NT;
    const int r = f >> 2, k4 = f & 3;
    const int ga = r0 + r, gb = c0 + r;
    ra[q] = ga < r_end ? __ldg(reinterpret_cast<const float4*>(Xc + (size_t)ga * Dp + k0) + k4)
                       : make_float4(0.f, 0.f, 0.f, 0.f);
    rb[q] = gb < c_end ? __ldg(reinterpret_cast<const float4*>(Xc + (size_t)gb * Dp + k0) + k4)
                       : make_float4(0.f, 0.f, 0.f, 0.f);
  }
}

__device__ __forceinline__ void store_stage(Stages& sm, int buf, int tid, const float4 (&ra)[2],
                                            const float4 (&rb)[2]) {
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    const int f = tid + q * NT;
    const int r = f >> 2, k4 = f & 3;
    sm.As[buf][4 * k4 + 0][r] = ra[q].x;
    sm.As[buf][4 * k4 + 1][r] = ra[q].y;
    sm.As[buf][4 * k4 + 2][r] = ra[q].z;
    sm.As[buf][4 * k4 + 3][r] = ra[q].w;
    sm.Bs[buf][4 * k4 + 0][r] = rb[q].x;
    sm.Bs[buf][4 * k4 + 1][r] = rb[q].y;
    sm.Bs[buf][4 * k4 + 2][r] = rb[q].z;
    sm.Bs[buf][4 * k4 + 3][r] = rb[q].w;
  }
}

// G rows [r0, r0+128) x columns [c0, c0+128) of the operand copy Xc (rows below `end`; the
// others count as zero) into g[row * pitch + column].
// Products are summed in partial sums of about sqrt(Dp) terms (whole stages) that
// then join the running sum: the rounding error of the two FP32 chains grows like
// sqrt(chain length), and two chains of about sqrt(Dp) terms each keep it smallest.
//
// 8 x 8 outputs per thread as packed FP32 pairs along the columns: a packed FMA does two
// FMAs in one issue slot (of two pipe cycles), which leaves slots for the shared-memory
// loads and for doubling the row operands. A warp covers 32 x 64 outputs (8 column and 4
// row positions), so that each of its four 16-byte operand loads per product reads at most
// 128 distinct bytes. One barrier per stage: the next stage is stored, and the one after
// requested, before this one is multiplied. 75 years, D = 3,726, L = 5, k = 20: 136.8 ms on
// both triangles with scalar FMAs, 60.3 ms now (0.63 of the FMA rate). What bounds it: a
// 16-byte shared-memory load of a warp takes four cycles of the SM's return path, so the
// four loads per product of eight warps take as long as their FMAs. 8 x 16 outputs per
// thread would need three quarters of that, but their partial sums leave no registers to hold
// the next operands (running sums in tensor memory, asynchronous copies: 67 to 81 ms).
__device__ __forceinline__ void gram_tile(Stages& sm, const float* __restrict__ Xc, int end,
                                          int Dp, int r0, int c0, int tid, float* g, int pitch) {
  const int lane = tid & 31, warp = tid >> 5;
  const int tx = (lane & 7) + 8 * (warp & 1), ty = (lane >> 3) + 4 * (warp >> 1);
  float2 acc[8][4], part[8][4];
#pragma unroll
  for (int i = 0; i < 8; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = part[i][j] = make_float2(0.f, 0.f);

  float4 ra[2], rb[2];
  const int nk = Dp / BK;
  const int flush = max(1, (int)(sqrtf((float)Dp) / BK + 0.5f));  // stages per partial sum
  load_stage(Xc, end, end, Dp, r0, c0, 0, tid, ra, rb);
  __syncthreads();  // previous users of the stages and of g are done
  store_stage(sm, 0, tid, ra, rb);
  if (nk > 1) load_stage(Xc, end, end, Dp, r0, c0, BK, tid, ra, rb);
  __syncthreads();
  int left = flush;  // stages until the partial sums join the running sums
  for (int kt = 0; kt < nk; ++kt) {
    const int cur = kt & 1;
    if (kt + 1 < nk) {
      store_stage(sm, cur ^ 1, tid, ra, rb);  // its readers passed the last barrier
      if (kt + 2 < nk) load_stage(Xc, end, end, Dp, r0, c0, (kt + 2) * BK, tid, ra, rb);
    }
#pragma unroll
    for (int kk = 0; kk < BK; ++kk) {
      const float4 a0 = *reinterpret_cast<const float4*>(&sm.As[cur][kk][ty * 4]);
      const float4 a1 = *reinterpret_cast<const float4*>(&sm.As[cur][kk][64 + ty * 4]);
      const float4 b0 = *reinterpret_cast<const float4*>(&sm.Bs[cur][kk][tx * 4]);
      const float4 b1 = *reinterpret_cast<const float4*>(&sm.Bs[cur][kk][64 + tx * 4]);
      const float av[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
      const float2 bv[4] = {make_float2(b0.x, b0.y), make_float2(b0.z, b0.w),
                            make_float2(b1.x, b1.y), make_float2(b1.z, b1.w)};
#pragma unroll
      for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j)
          part[i][j] = __ffma2_rn(make_float2(av[i], av[i]), bv[j], part[i][j]);
    }
    if (--left == 0 || kt + 1 == nk) {
      left = flush;
#pragma unroll
      for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          acc[i][j] = __fadd2_rn(acc[i][j], part[i][j]);
          part[i][j] = make_float2(0.f, 0.f);
        }
    }
    __syncthreads();
  }
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int r = (i < 4) ? ty * 4 + i : 64 + ty * 4 + (i - 4);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int c = (j < 2) ? tx * 4 + 2 * j : 64 + tx * 4 + 2 * (j - 2);
      g[r * pitch + c] = acc[i][j].x;
      g[r * pitch + c + 1] = acc[i][j].y;
    }
  }
  __syncthreads();
}

// ------------------------------------------------------- symmetric, shared work plan
struct Smem {
  Stages st;
  float G[BM][kPitch];          // kHalo carried columns, then the tile's 256
  float D[2][BM][kRowPitch];    // each group's rows of distances
  float W[2 * BN], T[2 * BN];   // window sums and bounds of the tile's output columns
  uint32_t finite[8];           // bit x of word ch: W[32 ch + x] is finite (candidate_masks)
  int cnt[2][64];               // column-side counters of each group
  WorkUnit unit;
};

// kBand: the band pre-pass (bounds only, no lists); S: shared minima per row.
template <bool kBand, int S>
__global__ void __launch_bounds__(NT, 1)
    fused_fp32_kernel(const float* __restrict__ Xc, const __grid_constant__ TcArgs a,
                      const __grid_constant__ TcWork w, const __grid_constant__ SeriesTable sr) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  Smem& sm = *reinterpret_cast<Smem*>(smem_raw);
  const int tid = threadIdx.x;
  const int gid = tid >> 7, l = tid & 127, bar = 1 + gid;  // group, row, named barrier
  ColSide cs;
  cs.cnt = sm.cnt[gid];
  cs.turn = 0;
  if (l < 64) cs.cnt[l] = 0;
  float* drow = sm.D[gid][l];
  unsigned cnt[5] = {0, 0, 0, 0, 0};
  launch_wait();
  launch_next();
  for (;;) {
    __syncthreads();  // the last unit's readers are done
    if (tid == 0) {
      const int u = atomicAdd(w.counter, 1);
      if (u < w.nunits) sm.unit = w.units[u];
      else sm.unit.strip = -1;
    }
    __syncthreads();
    const WorkUnit wu = sm.unit;
    if (wu.strip < 0) break;
    UnitSpan us;
    if (!unit_span(wu, sr.s, 0, us)) continue;
    const int nser = us.nser, ntiles = us.ntiles;
    const int rows_end = us.row_base + us.M + us.L - 1;  // day rows of the (first) series
    RowSide rs;
    GroupMin<false> gm;
    rs.reset();
    gm.reset();
    for (int it = 0; it < ntiles; ++it) {
      const int c0 = us.jlo + it * us.adv;
#pragma unroll 1
      for (int half = 0; half < 2; ++half)  // (the second only where an output needs it)
        if (half == 0 || c0 + BN < us.jhi + a.Lmax - 1)
          gram_tile(sm.st, Xc, rows_end, a.Dp, us.row_base + us.T0,
                    us.row_base + c0 + half * BN, tid, &sm.G[0][kHalo + half * BN], kPitch);
      for (int sj = 0; sj < nser; ++sj) {
        if (nser > 1) {
          unit_span(wu, sr.s, sj, us);
          if (sj > 0) __syncthreads();  // W, T and the second group's minima have been read
        }
        const int L = us.L, t = us.T0 + l;
        const bool row_ok = l < us.R && t < us.M;
        const float Wt = row_ok ? a.W[us.out_base + t] : 0.f;
        float thr_row = row_ok ? __uint_as_float(__ldcg(w.thr + us.out_base + t)) : 0.f;
        if (nser > 1 || it == 0) {
          rs.reset();
          gm.reset();
          if (!kBand)
            rs.rec = a.part +
                     (size_t)(us.part_base + (long long)t * us.slots + us.slot * 2 + gid) * a.cap;
        }
        {
          const int j = c0 - (L - 1) + tid;
          const bool in = j >= 0 && j < us.M;
          const float wj = in ? a.W[us.out_base + j] : 0.f;
          sm.W[tid] = wj;
          const uint32_t f = __ballot_sync(0xffffffffu, wj < CUDART_INF_F);
          if ((tid & 31) == 0) sm.finite[tid >> 5] = f;
          sm.T[tid] = in ? __uint_as_float(__ldcg(w.thr + us.out_base + j)) : 0.f;
        }
        const int jsym = us.T0 + us.R;  // column side from here on (sym)
        const long long cbase = w.sym ? us.col_base + w.col_off[us.strip_base + us.strip] : 0;
        __syncthreads();
#pragma unroll 1
        for (int ch = 4 * gid; ch < 4 * gid + 4; ++ch) {
          // output columns j0 + x, whose windows start in G column kHalo - (L-1) + 32 ch + x;
          // the first L-1 columns of a unit's first chunk have no carried window
          const int j0 = c0 + ch * 32 - (L - 1);
          const int xfirst = (ch == 0 && (it == 0 || !us.carry)) ? L - 1 : 0;
          const uint32_t unitrange = bit_range(xfirst, 32) & bit_range(us.jlo - j0, us.jhi - j0);
          if (unitrange == 0) continue;  // the same for the whole group
          const uint32_t colrange = w.sym ? bit_range(jsym - j0, 32) & unitrange : 0u;
          uint32_t cand = 0, ccand = 0;
          float c[32];
          if (row_ok && Wt < CUDART_INF_F) {
            const float* g = &sm.G[l][kHalo - (L - 1) + ch * 32];
#pragma unroll
            for (int x = 0; x < 32; ++x) c[x] = g[x];
            for (int m = 1; m < L; ++m) {
              const float* gmx = g + m * (kPitch + 1);
#pragma unroll
              for (int x = 0; x < 32; ++x) c[x] += gmx[x];
            }
            distances(c, Wt, sm.W + ch * 32, 0.f);
            const uint32_t valid = unitrange & sm.finite[ch] & ~bit_range(t - us.e - j0, t + us.e + 1 - j0);
            if (kBand) {
              gm.scan(c, valid);
            } else {
              candidate_masks(c, rs.limit(thr_row), sm.T + ch * 32, cand, ccand);
              cand &= valid;
              ccand &= valid & colrange;
            }
          }
          if (!kBand) {
            const uint32_t cmask = ccand;
            if (cand | ccand) store_row<true>(drow, c);
            cnt[0] += __popc(cand);
            cnt[1] += __popc(ccand);
            const bool over = append<S>(rs, cs, cand, ccand, drow, j0, us.k, t,
                                        cbase + (j0 - jsym), a.shared_min + us.out_base + t,
                                        a.shared_min + us.out_base + j0, w, a);
            if (colrange) {
              const int ne = cs.finish<true>(over, colrange, cmask, c, &sm.D[gid][0][0],
                                             kRowPitch, l, l, bar, us.k, us.T0, us.strip,
                                             us.out_base, j0, cbase + (j0 - jsym), w, a);
              cnt[3] += ne > 0;
              cnt[2] += ne > us.k;
            }
            rs.compress(us.k, a, w.thr + us.out_base + t);
          }
          cnt[4] += l == 0;
        }
        const bool last = nser > 1 || it == ntiles - 1;
        if (kBand && last) {
          // the second group hands its minima to the first
          float* xb = &sm.D[1][0][0];
          if (gid == 1)
#pragma unroll
            for (int x = 0; x < 32; ++x) xb[x * BM + l] = gm.m[x];
          __syncthreads();
          if (gid == 0) {
            const float bd = gm.bound(us.k, xb + l);
            if (row_ok && bd < thr_row && tk_in(us.out_base + t, a.out_rows, a.err))
              publish_bound(w.thr + us.out_base + t, bd);
          }
        } else if (!kBand && (last || (it + 1) % a.bound_tiles == 0)) {
          const float bd = row_bound<S>(us.k, a.shared_min + us.out_base + t, a.out_rows, row_ok,
                                        thr_row);
          if (row_ok && bd < thr_row && tk_in(us.out_base + t, a.out_rows, a.err))
            publish_bound(w.thr + us.out_base + t, bd);
        }
        if (!kBand && last && row_ok && us.jlo < us.jhi) {
          const long long li = us.part_base + (long long)t * us.slots + us.slot * 2 + gid;
          if (tk_in(li, w.part_lists, a.err)) a.part_n[li] = rs.n;
        }
      }
      if (nser > 1) unit_span(wu, sr.s, 0, us);
      __syncthreads();
      if (us.carry && it + 1 < ntiles) {
        const int L = us.L;
        for (int q = tid; q < BM * (L - 1); q += NT) {
          const int r = q / (L - 1), c = q - r * (L - 1);
          sm.G[r][kHalo - (L - 1) + c] = sm.G[r][kHalo + 2 * BN - (L - 1) + c];
        }
      }
    }
  }
  if (w.stats) {
#pragma unroll
    for (int i = 0; i < 5; ++i) {
      const unsigned v = __reduce_add_sync(0xffffffffu, cnt[i]);
      if ((tid & 31) == 0 && v) atomicAdd(w.stats + kStatRowInserts + i, (unsigned long long)v);
    }
  }
}

// ------------------------------------------------------------- both triangles
struct SmemBoth {
  Stages st;
  float G[BM][kPitchBoth];
};

__global__ void __launch_bounds__(NT, 1)
    fused_fp32_both_kernel(const float* __restrict__ Xc, FusedArgs a) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  SmemBoth& sm = *reinterpret_cast<SmemBoth*>(smem_raw);
  const Schedule& s = a.sch;
  SmemList list;
  list.d = reinterpret_cast<float*>(smem_raw + sizeof(SmemBoth));
  list.i = reinterpret_cast<int32_t*>(list.d + BM * s.k);
  list.stride = BM;
  list.k = s.k;

  const int tid = threadIdx.x;
  const int L = s.L;
  launch_wait();
  launch_next();
  for (int u = blockIdx.x; u < s.units; u += gridDim.x) {
    const UnitCoord uc = unit_coord(s, u);
    if (uc.strip >= s.strips) continue;
    RowCtx rc;
    rc.L = L;
    rc.e = s.e;
    rc.jlo = uc.chunk * s.chunk_cols;
    rc.jhi = min(s.M, rc.jlo + s.chunk_cols);
    if (rc.jlo >= rc.jhi) continue;
    const int T0 = uc.strip * s.rows_out;
    rc.lrow = tid;
    rc.t = T0 + tid;
    const bool row_ok = tid < s.rows_out && rc.t < s.M;
    rc.Wt = row_ok ? a.W[rc.t] : 0.f;
    float thr = CUDART_INF_F;
    if (tid < BM) list.reset(tid);

    const int ntiles = (rc.jhi - rc.jlo + L - 1 + BN - 1) / BN;
    for (int it = 0; it < ntiles; ++it) {
      const int c0 = rc.jlo + it * BN;  // first Gram column of the tile
      gram_tile(sm.st, Xc, a.N, a.Dp, T0, c0, tid, &sm.G[0][kHalo], kPitchBoth);
      // output column x of this tile is j = c0 - (L-1) + x; its window starts in
      // the carried columns, which sit just left of kHalo
      if (row_ok)
        window_topk(&sm.G[0][kHalo - (L - 1)], kPitchBoth, rc, it == 0 ? L - 1 : 0, BN,
                    c0 - (L - 1), a.W, list, tid, thr);
      __syncthreads();
      for (int q = tid; q < BM * (L - 1); q += NT) {
        const int r = q / (L - 1), c = q - r * (L - 1);
        sm.G[r][kHalo - (L - 1) + c] = sm.G[r][kHalo + BN - (L - 1) + c];
      }
    }
    if (row_ok) {
      const size_t base = ((size_t)rc.t * s.chunks + uc.chunk) * s.k;
      for (int p = 0; p < s.k; ++p) {
        a.part_d[base + p] = list.d[p * BM + tid];
        a.part_i[base + p] = list.i[p * BM + tid];
      }
    }
  }
}

template <bool kBand, int S>
cudaError_t launch_sym(const float* Xc, const TcArgs& a, const TcWork& w, const SeriesTable& sr,
                       int num_ctas, cudaStream_t st) {
  cudaError_t err =
      cudaFuncSetAttribute(fused_fp32_kernel<kBand, S>,
                           cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(Smem));
  if (err != cudaSuccess) return err;
  return launch_chained(fused_fp32_kernel<kBand, S>, num_ctas, NT, sizeof(Smem), st, Xc, a, w, sr);
}

}  // namespace

cudaError_t launch_fused_fp32(const float* Xc, const TcArgs& a, const TcWork& w,
                              const SeriesTable& sr, int num_ctas, cudaStream_t st) {
  if (!w.write_lists) return launch_sym<true, 64>(Xc, a, w, sr, num_ctas, st);
  return min_slots(a.kmax) == 64 ? launch_sym<false, 64>(Xc, a, w, sr, num_ctas, st)
                                 : launch_sym<false, 128>(Xc, a, w, sr, num_ctas, st);
}

cudaError_t launch_fused_fp32_both(const float* Xc, const FusedArgs& a, int num_ctas,
                                     cudaStream_t st) {
  const size_t smem = sizeof(SmemBoth) + (size_t)BM * a.sch.k * 8;
  cudaError_t err = cudaFuncSetAttribute(fused_fp32_both_kernel,
                                         cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (err != cudaSuccess) return err;
  return launch_chained(fused_fp32_both_kernel, num_ctas, NT, smem, st, Xc, a);
}

}  // namespace traknn
