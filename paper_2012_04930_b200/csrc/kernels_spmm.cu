// Y = epi(A X) for a CSR matrix A and a row-major fp32 matrix X: the normalized
// adjacency product of the GCN layer (Section 4.1) and, over the transposed
// CSR, of its backward pass.
//
// One warp per row, rows issued longest class first (the caller's degree-sorted
// permutation); the first n_long rows of that permutation (hub rows of a
// power-law graph) get a whole thread block each.  The 32 lanes form 32 / G groups of G lanes; every group owns a
// contiguous slice of the row's non-zeros and every lane CH float4 column
// chunks, so one warp instruction gathers 32 / G feature rows with 16 bytes per
// lane.  With G < 32 column indices and values are read four at a time with
// 16-byte loads whose address is the same for all lanes of a group, U such quads
// ahead of the gathers; with G = 32 and stored values they are fetched coalesced,
// 32 at a time, and handed round through 128-byte slots of shared memory per warp.
// Each output row has one writer and a fixed summation order: no atomics,
// bitwise reproducible.
#include <cuda_runtime.h>

#include <algorithm>

#include "debug_check.h"
#include "internal.h"
#include "launch.h"

namespace gcnsa {

namespace {

constexpr unsigned kFull = 0xffffffffu;

#if GCNSA_DBG
GCNSA_DBG_WORD(g_dbg_spmm);
// a gathered column index must name a row of the source matrix
#define GCNSA_CHECK_COLUMN(cc) \
  if (dbg.src_rows >= 0 && !dbg_in(&g_dbg_spmm, (cc), 0, dbg.src_rows, kDbgColumn)) return
// the bounds travel as an extra (by-value) parameter of the checking build's kernels and device functions
#define GCNSA_DBG_PARAM , const SpmmBounds dbg
#define GCNSA_DBG_ARG , dbg
#define GCNSA_DBG_LAUNCH_ARG , a.dbg
#else
#define GCNSA_CHECK_COLUMN(cc)
#define GCNSA_DBG_PARAM
#define GCNSA_DBG_ARG
#define GCNSA_DBG_LAUNCH_ARG
#endif

__device__ __forceinline__ void fma4(float4& acc, float a, const float4& x) {
  acc.x = fmaf(a, x.x, acc.x);
  acc.y = fmaf(a, x.y, acc.y);
  acc.z = fmaf(a, x.z, acc.z);
  acc.w = fmaf(a, x.w, acc.w);
}

__device__ __forceinline__ void add4(float4& acc, const float4& x) {
  acc.x += x.x;
  acc.y += x.y;
  acc.z += x.z;
  acc.w += x.w;
}

// Adds the non-zeros [beg, end) that fall into slice `slice` of `n_slices` equal quad ranges to acc.
// UNIT: every stored entry counts as 1 (the 0/1 pattern A + I); `val` is not read.
template <int G, int CH, int U, bool UNIT>
__device__ __forceinline__ void accumulate_slice(float4 (&acc)[CH], int beg, int end, int slice, int n_slices, int gl,
                                                 const int32_t* __restrict__ col, const float* __restrict__ val,
                                                 const float4* __restrict__ x, int64_t ldx4, int nvec, int vec_idx GCNSA_DBG_PARAM) {
  const float4* xl = x + gl;
  auto gather = [&](int cc, float vv) {
    GCNSA_CHECK_COLUMN(cc);
    const float4* xr = xl + (int64_t)cc * ldx4;
#pragma unroll
    for (int ch = 0; ch < CH; ++ch)
      if (gl + ch * G < nvec) {
        if (UNIT) add4(acc[ch], __ldg(xr + ch * G));
        else fma4(acc[ch], vv, __ldg(xr + ch * G));
      }
  };
  auto edge_quad = [&](int e0) {  // a quad that sticks out of [beg, end): element by element
    for (int t = 0; t < 4; ++t) {
      const int e = e0 + t;
      if (e >= beg && e < end) gather(__ldg(col + e), UNIT ? 1.f : __ldg(val + e));
    }
  };
  // quads are aligned to absolute multiples of 4 so that their loads are 16-byte aligned
  const int a0 = beg & ~3;
  const int nq = (end - a0 + 3) >> 2;
  const int qps = (nq + n_slices - 1) / n_slices;
  const int q0 = slice * qps, q1 = min(nq, q0 + qps);
  int q = q0;
  if (q < q1 && a0 + 4 * q < beg) {
    edge_quad(a0 + 4 * q);
    ++q;
  }
  const int qfull = vec_idx ? min(q1, (end - a0) >> 2) : q;  // quads that lie entirely below `end`
  for (; q + U <= qfull; q += U) {
    int4 c4[U];
    float4 v4[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      c4[u] = __ldg(reinterpret_cast<const int4*>(col + a0 + 4 * (q + u)));
      if (!UNIT) v4[u] = __ldg(reinterpret_cast<const float4*>(val + a0 + 4 * (q + u)));
      else v4[u] = make_float4(1.f, 1.f, 1.f, 1.f);
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      gather(c4[u].x, v4[u].x);
      gather(c4[u].y, v4[u].y);
      gather(c4[u].z, v4[u].z);
      gather(c4[u].w, v4[u].w);
    }
  }
  for (; q < qfull; ++q) {
    const int4 c4 = __ldg(reinterpret_cast<const int4*>(col + a0 + 4 * q));
    const float4 v4 = UNIT ? make_float4(1.f, 1.f, 1.f, 1.f) : __ldg(reinterpret_cast<const float4*>(val + a0 + 4 * q));
    gather(c4.x, v4.x);
    gather(c4.y, v4.y);
    gather(c4.z, v4.z);
    gather(c4.w, v4.w);
  }
  for (; q < q1; ++q) edge_quad(a0 + 4 * q);
}

// The element range of slice `slice` of `n_slices` (the same cut into aligned quads as accumulate_slice makes).
__device__ __forceinline__ void slice_range(int beg, int end, int slice, int n_slices, int& e0, int& e1) {
  const int a0 = beg & ~3;
  const int nq = (end - a0 + 3) >> 2;
  const int qps = (nq + n_slices - 1) / n_slices;
  const int q0 = slice * qps, q1 = min(nq, q0 + qps);
  e0 = max(beg, a0 + 4 * q0);
  e1 = q0 < q1 ? min(end, a0 + 4 * q1) : e0;
}

// Whole-warp shapes (G = 32: every lane holds CH chunks of the same source row) that read stored values.  A
// warp-uniform 16-byte load of four indices or values costs the L1 data path four wavefronts, one per non-zero,
// next to the four of a 512-byte gather.  Here lane l fetches the index and value of non-zero base + l, one
// coalesced wavefront per 32 non-zeros, the warp parks them in its 128-byte slots of shared memory and reads them
// back four at a time as broadcasts; the fetch of the next 32 is in flight while the current 32 are gathered.
// Elements are added in index order, as in accumulate_slice.  (With unit entries only the indices are left to
// broadcast; there the uniform loads of accumulate_slice measured 1 % faster, so that path keeps them.)
template <int CH, bool UNIT>
__device__ __forceinline__ void accumulate_range_staged(float4 (&acc)[CH], int e0, int e1, int lane,
                                                        const int32_t* __restrict__ col, const float* __restrict__ val,
                                                        const float4* __restrict__ x, int64_t ldx4, int nvec,
                                                        int32_t* sidx, float* sval GCNSA_DBG_PARAM) {
  const float4* xl = x + lane;
  auto gather = [&](int cc, float vv) {
    GCNSA_CHECK_COLUMN(cc);
    const float4* xr = xl + (int64_t)cc * ldx4;
#pragma unroll
    for (int ch = 0; ch < CH; ++ch)
      if (lane + ch * 32 < nvec) {
        if (UNIT) add4(acc[ch], __ldg(xr + ch * 32));
        else fma4(acc[ch], vv, __ldg(xr + ch * 32));
      }
  };
  int nxt_c = 0;
  float nxt_v = 0.f;
  if (e0 + lane < e1) {
    nxt_c = __ldg(col + e0 + lane);
    if (!UNIT) nxt_v = __ldg(val + e0 + lane);
  }
  for (int base = e0; base < e1; base += 32) {
    __syncwarp();  // the reads of the previous 32 are done
    sidx[lane] = nxt_c;
    if (!UNIT) sval[lane] = nxt_v;
    __syncwarp();
    if (base + 32 + lane < e1) {
      nxt_c = __ldg(col + base + 32 + lane);
      if (!UNIT) nxt_v = __ldg(val + base + 32 + lane);
    }
    const int cnt = min(32, e1 - base);
    int k = 0;
#pragma unroll 4
    for (; k + 4 <= cnt; k += 4) {
      const int4 c4 = *reinterpret_cast<const int4*>(sidx + k);
      float4 v4 = make_float4(1.f, 1.f, 1.f, 1.f);
      if (!UNIT) v4 = *reinterpret_cast<const float4*>(sval + k);
      gather(c4.x, v4.x);
      gather(c4.y, v4.y);
      gather(c4.z, v4.z);
      gather(c4.w, v4.w);
    }
    for (; k < cnt; ++k) gather(sidx[k], UNIT ? 1.f : sval[k]);
  }
}

// Folds the 32 / G group sums of a warp (fixed order); afterwards the lanes of group 0 hold the warp's sum.
template <int G, int CH>
__device__ __forceinline__ void fold_groups(float4 (&acc)[CH]) {
#pragma unroll
  for (int off = G; off < 32; off <<= 1) {
#pragma unroll
    for (int ch = 0; ch < CH; ++ch) {
      acc[ch].x += __shfl_xor_sync(kFull, acc[ch].x, off);
      acc[ch].y += __shfl_xor_sync(kFull, acc[ch].y, off);
      acc[ch].z += __shfl_xor_sync(kFull, acc[ch].z, off);
      acc[ch].w += __shfl_xor_sync(kFull, acc[ch].w, off);
    }
  }
}

// Epilogue + store of float4 chunk qq of one output row.
__device__ __forceinline__ void store_chunk(float4 r, int row, int qq, int f, int epi, const float* __restrict__ aux,
                                            int64_t ldaux, float* __restrict__ y, int64_t ldy) {
  const int c0 = qq * 4;
  if (epi == GCNSA_EPI_BIAS || epi == GCNSA_EPI_BIAS_RELU) {
    if (aux) {
      r.x += (c0 + 0 < f) ? __ldg(aux + c0 + 0) : 0.f;
      r.y += (c0 + 1 < f) ? __ldg(aux + c0 + 1) : 0.f;
      r.z += (c0 + 2 < f) ? __ldg(aux + c0 + 2) : 0.f;
      r.w += (c0 + 3 < f) ? __ldg(aux + c0 + 3) : 0.f;
    }
    if (epi == GCNSA_EPI_BIAS_RELU) {
      r.x = fmaxf(r.x, 0.f);
      r.y = fmaxf(r.y, 0.f);
      r.z = fmaxf(r.z, 0.f);
      r.w = fmaxf(r.w, 0.f);
    }
  } else if (epi == GCNSA_EPI_MASK) {
    const float4 mk = __ldg(reinterpret_cast<const float4*>(aux + (int64_t)row * ldaux) + qq);
    r.x = mk.x > 0.f ? r.x : 0.f;
    r.y = mk.y > 0.f ? r.y : 0.f;
    r.z = mk.z > 0.f ? r.z : 0.f;
    r.w = mk.w > 0.f ? r.w : 0.f;
  }
  reinterpret_cast<float4*>(y + (int64_t)row * ldy)[qq] = r;
}

// Rows of a few dozen entries (33 in the degree-32 random graph, 20 in the block models, four fifths of the rows of the
// 2.45 M-vertex graph): with a warp per row the loads that depend on one another (order, row pointers, indices, rows) and
// the folding of the groups' sums outweigh the gathers.  Here a group of G lanes owns a row, every lane CH float4 chunks
// of it, so a warp works on 32 / G rows of one length class at a time and nothing is folded.  A group fetches the indices
// of 16 (G < 16) or G entries with coalesced loads, the next ones while these are gathered, and hands them round by
// shuffle; U gathers per lane are in flight.  w: the group's place in the processing order.
template <int G, int CH, int U, bool UNIT>
__device__ __forceinline__ void short_rows(int w, int n_rows, const int32_t* __restrict__ rowptr, const int32_t* __restrict__ col,
                                           const float* __restrict__ val, const float* __restrict__ rscale,
                                           const int32_t* __restrict__ order, const float4* __restrict__ x, int64_t ldx4, int nvec,
                                           int f, int epi, const float* __restrict__ aux, int64_t ldaux, float* __restrict__ y,
                                           int64_t ldy GCNSA_DBG_PARAM) {
  constexpr int B = G < 16 ? 16 : G, L = B / G;  // entries per round, indices per lane
  const int gl = threadIdx.x % G;
  bool ok = w < n_rows;
  if (!__any_sync(kFull, ok)) return;
  int row = 0, beg = 0, n = 0;
  if (ok) {
    row = __ldg(order + w);
#if GCNSA_DBG
    ok = dbg.mat_rows < 0 || dbg_in(&g_dbg_spmm, row, 0, dbg.mat_rows, kDbgOrderEntry);
#endif
  }
  if (ok) {
    beg = __ldg(rowptr + row);
    const int end = __ldg(rowptr + row + 1);
#if GCNSA_DBG
    ok = dbg_in(&g_dbg_spmm, beg, 0, (long long)end + 1, kDbgRowRange) &&
         (dbg.nnz < 0 || dbg_in(&g_dbg_spmm, end, 0, dbg.nnz + 1, kDbgRowRange));
#endif
    if (ok) n = end - beg;
  }
  const int n_max = __reduce_max_sync(kFull, n);
  float4 acc[CH];
#pragma unroll
  for (int ch = 0; ch < CH; ++ch) acc[ch] = make_float4(0.f, 0.f, 0.f, 0.f);
  int nxt[L];
  float nxt_v[L];
  auto fetch = [&](int base) {
#pragma unroll
    for (int j = 0; j < L; ++j) {
      const int k = base + j * G + gl;
      nxt[j] = k < n ? __ldg(col + beg + k) : 0;
      nxt_v[j] = !UNIT && k < n ? __ldg(val + beg + k) : 0.f;
    }
  };
  fetch(0);
  for (int base = 0; base < n_max; base += B) {
    int mine[L];
    float wgt[L];
#pragma unroll
    for (int j = 0; j < L; ++j) { mine[j] = nxt[j]; wgt[j] = nxt_v[j]; }
    if (base + B < n_max) fetch(base + B);
#pragma unroll
    for (int k0 = 0; k0 < B; k0 += U) {
      if (base + k0 >= n_max) break;  // all rows of the warp alike
      float4 v[U][CH];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int k = k0 + u;
        const int c = __shfl_sync(kFull, mine[k / G], k % G, G);
        bool live = base + k < n;
#if GCNSA_DBG
        if (live && dbg.src_rows >= 0) live = dbg_in(&g_dbg_spmm, c, 0, dbg.src_rows, kDbgColumn);
#endif
        const float4* xr = x + (int64_t)c * ldx4 + gl;
#pragma unroll
        for (int ch = 0; ch < CH; ++ch)
          v[u][ch] = live && gl + ch * G < nvec ? __ldg(xr + ch * G) : make_float4(0.f, 0.f, 0.f, 0.f);
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int k = k0 + u;
        const float sv = UNIT ? 1.f : __shfl_sync(kFull, wgt[k / G], k % G, G);
#pragma unroll
        for (int ch = 0; ch < CH; ++ch) {
          if (UNIT) add4(acc[ch], v[u][ch]);
          else fma4(acc[ch], sv, v[u][ch]);
        }
      }
    }
  }
  if (!ok) return;
  const float sc = rscale ? __ldg(rscale + row) : 1.f;
#pragma unroll
  for (int ch = 0; ch < CH; ++ch) {
    const int qq = gl + ch * G;
    if (qq >= nvec) continue;
    float4 r = acc[ch];
    if (rscale) { r.x *= sc; r.y *= sc; r.z *= sc; r.w *= sc; }
    store_chunk(r, row, qq, f, epi, aux, ldaux, y, ldy);
  }
}

// Blocks [0, n_long): one thread block per long row order[b]; its TPB / 32 warps take equal parts of the row,
// their sums meet in shared memory and are added in warp order (fixed order), so a hub row of thousands of
// non-zeros is not one warp's serial chain.  Blocks after that: one warp per row order[n_long .. n_warp), then a group of
// lanes per row order[n_warp .. n_rows) (short_rows<SG, SCH, SU>).  One launch, longest rows dispatched first.
template <int G, int CH, int U, int TPB, int MINB, bool UNIT, int SG, int SCH, int SU>
__global__ void __launch_bounds__(TPB, MINB)
spmm_rows(int n_long, int n_warp, int n_rows, const int32_t* __restrict__ rowptr, const int32_t* __restrict__ col,
          const float* __restrict__ val, const float* __restrict__ rscale, const int32_t* __restrict__ order,
          const float4* __restrict__ x, int64_t ldx4,
          int nvec, int f, int vec_idx, int epi, const float* __restrict__ aux, int64_t ldaux, float* __restrict__ y,
          int64_t ldy GCNSA_DBG_PARAM) {
  wait_for_predecessors();
  constexpr int NG = 32 / G;
  constexpr int W = TPB / 32;
  __shared__ float4 part[W][G * CH];
  __shared__ __align__(16) int32_t stage_idx[(G == 32 && !UNIT) ? W : 1][32];
  __shared__ __align__(16) float stage_val[(G == 32 && !UNIT) ? W : 1][32];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int g = lane / G, gl = lane % G;
  float4 acc[CH];
#pragma unroll
  for (int ch = 0; ch < CH; ++ch) acc[ch] = make_float4(0.f, 0.f, 0.f, 0.f);

  if ((int)blockIdx.x < n_long) {
    const int row = __ldg(order + blockIdx.x);
#if GCNSA_DBG
    if (dbg.mat_rows >= 0 && !dbg_in(&g_dbg_spmm, row, 0, dbg.mat_rows, kDbgOrderEntry)) return;  // whole block alike
#endif
    const int beg = __ldg(rowptr + row), end = __ldg(rowptr + row + 1);
#if GCNSA_DBG
    if (!dbg_in(&g_dbg_spmm, beg, 0, (long long)end + 1, kDbgRowRange)) return;
    if (dbg.nnz >= 0 && !dbg_in(&g_dbg_spmm, end, 0, dbg.nnz + 1, kDbgRowRange)) return;
#endif
    if constexpr (G == 32 && !UNIT) {
      int e0, e1;
      slice_range(beg, end, warp, W, e0, e1);
      accumulate_range_staged<CH, UNIT>(acc, e0, e1, lane, col, val, x, ldx4, nvec, stage_idx[warp], stage_val[warp] GCNSA_DBG_ARG);
    } else {
      accumulate_slice<G, CH, U, UNIT>(acc, beg, end, warp * NG + g, W * NG, gl, col, val, x, ldx4, nvec, vec_idx GCNSA_DBG_ARG);
    }
    fold_groups<G, CH>(acc);
    if (g == 0) {
#pragma unroll
      for (int ch = 0; ch < CH; ++ch) part[warp][gl + ch * G] = acc[ch];
    }
    __syncthreads();
    if (warp != 0 || g != 0) return;
#pragma unroll
    for (int ch = 0; ch < CH; ++ch) {
      const int qq = gl + ch * G;
      if (qq >= nvec) continue;
      float4 r = part[0][qq];
#pragma unroll
      for (int k = 1; k < W; ++k) {
        const float4 t = part[k][qq];
        r.x += t.x; r.y += t.y; r.z += t.z; r.w += t.w;
      }
      if (rscale) {
        const float sc = __ldg(rscale + row);
        r.x *= sc; r.y *= sc; r.z *= sc; r.w *= sc;
      }
      store_chunk(r, row, qq, f, epi, aux, ldaux, y, ldy);
    }
    return;
  }
  const int b = (int)blockIdx.x - n_long, b_short = b - (n_warp - n_long + W - 1) / W;
  if (b_short >= 0) {
    short_rows<SG, SCH, SU, UNIT>(n_warp + (b_short * W + warp) * (32 / SG) + lane / SG, n_rows, rowptr, col, val, rscale, order, x,
                                  ldx4, nvec, f, epi, aux, ldaux, y, ldy GCNSA_DBG_ARG);
    return;
  }
  const int w = n_long + b * W + warp;
  if (w >= n_warp) return;
  const int row = order ? __ldg(order + w) : w;
#if GCNSA_DBG
  if (dbg.mat_rows >= 0 && !dbg_in(&g_dbg_spmm, row, 0, dbg.mat_rows, kDbgOrderEntry)) return;  // whole warp alike
#endif
  const int beg = __ldg(rowptr + row), end = __ldg(rowptr + row + 1);
#if GCNSA_DBG
  if (!dbg_in(&g_dbg_spmm, beg, 0, (long long)end + 1, kDbgRowRange)) return;
  if (dbg.nnz >= 0 && !dbg_in(&g_dbg_spmm, end, 0, dbg.nnz + 1, kDbgRowRange)) return;
#endif
  if constexpr (G == 32 && !UNIT) {
    accumulate_range_staged<CH, UNIT>(acc, beg, end, lane, col, val, x, ldx4, nvec, stage_idx[warp], stage_val[warp] GCNSA_DBG_ARG);
  } else {
    accumulate_slice<G, CH, U, UNIT>(acc, beg, end, g, NG, gl, col, val, x, ldx4, nvec, vec_idx GCNSA_DBG_ARG);
  }
  fold_groups<G, CH>(acc);
  if (g != 0) return;
  const float sc = rscale ? __ldg(rscale + row) : 1.f;
#pragma unroll
  for (int ch = 0; ch < CH; ++ch) {
    const int qq = gl + ch * G;
    if (qq >= nvec) continue;
    float4 r = acc[ch];
    if (rscale) { r.x *= sc; r.y *= sc; r.z *= sc; r.w *= sc; }
    store_chunk(r, row, qq, f, epi, aux, ldaux, y, ldy);
  }
}

struct Args {
  cudaStream_t s;
  int n_rows;
  const int32_t *rowptr, *col;
  const float* val;
  const float* rscale;
  const int32_t* order;
  int n_long, n_warp;
  const float* x;
  int64_t ldx;
  int nvec, f, vec_idx, epi;
  const float* aux;
  int64_t ldaux;
  float* y;
  int64_t ldy;
  SpmmBounds dbg;
};

template <int G, int CH, int U, int TPB, int MINB, int SG, int SCH, int SU>
cudaError_t run(const Args& a) {
  const int rows_per_block = TPB / 32, short_per_block = rows_per_block * (32 / SG);
  const int grid = a.n_long + (a.n_warp - a.n_long + rows_per_block - 1) / rows_per_block +
                   (a.n_rows - a.n_warp + short_per_block - 1) / short_per_block;
  if (a.val)
    launch(spmm_rows<G, CH, U, TPB, MINB, false, SG, SCH, SU>, grid, TPB, 0, a.s,
        a.n_long, a.n_warp, a.n_rows, a.rowptr, a.col, a.val, a.rscale, a.order, reinterpret_cast<const float4*>(a.x), a.ldx / 4,
        a.nvec, a.f, a.vec_idx, a.epi, a.aux, a.ldaux, a.y, a.ldy GCNSA_DBG_LAUNCH_ARG);
  else
    launch(spmm_rows<G, CH, U, TPB, MINB, true, SG, SCH, SU>, grid, TPB, 0, a.s,
        a.n_long, a.n_warp, a.n_rows, a.rowptr, a.col, nullptr, a.rscale, a.order, reinterpret_cast<const float4*>(a.x), a.ldx / 4,
        a.nvec, a.f, a.vec_idx, a.epi, a.aux, a.ldaux, a.y, a.ldy GCNSA_DBG_LAUNCH_ARG);
  note_launch();
  return cudaGetLastError();
}

// ---- the remainder of a planned product ------------------------------------------------------------------------
// Row = its partial sums from the tensor-core kernel plus its entries [rowptr, rowend) of the remainder CSR (SCALED:
// each times the scale of its source row), then the epilogue of spmm_rows.  A row has few entries here (a few
// per cent of its own on the 233 K-vertex graph), so what counts is the chain of dependent loads as much as the gathers: the warp fetches 32 indices with one load and hands them round by shuffle, RU gathers per group are in flight
// at once, and the partial sums are asked for before the first gather.
template <int CH>
__device__ __forceinline__ void load_pieces(float4 (&out)[CH], const SpmmBase& b, int row, int q_first, int q_step, int nvec) {
  const int pos = __ldg(b.pos + row), t = pos / kDenseRows, w4 = b.width / 4;
  const int first = __ldg(b.prefix + t), cnt = __ldg(b.prefix + t + 1) - first;
#pragma unroll
  for (int ch = 0; ch < CH; ++ch) {
    out[ch] = make_float4(0.f, 0.f, 0.f, 0.f);
    const int qq = q_first + ch * q_step;
    if (cnt == 0 || qq >= nvec) continue;
    const int Q = b.q0 + qq, slab = b.nslab > 1 ? Q / w4 : 0;
    const unsigned u0 = b.nslab * first + slab * cnt, u1 = u0 + cnt - 1;
    const int c0 = b.magic ? __umulhi(u0, b.magic) : u0 / b.per_cta, c1 = b.magic ? __umulhi(u1, b.magic) : u1 / b.per_cta;
#if GCNSA_DBG
    if (!dbg_in(&g_dbg_spmm, (long long)t * b.nslab + slab + c1, t * b.nslab + slab + c0, b.n_pieces, kDbgPartialSum)) continue;
#endif
    const float4* src = reinterpret_cast<const float4*>(b.pieces) +
                        ((int64_t)(t * b.nslab + slab + c0) * kDenseRows + (pos % kDenseRows)) * w4 + (Q - slab * w4);
    out[ch] = __ldg(src);
    for (int c = c0 + 1; c <= c1; ++c) {
      src += (int64_t)kDenseRows * w4;
      add4(out[ch], __ldg(src));
    }
  }
}

template <int G, int CH, int RU, bool SCALED>
__device__ __forceinline__ void gather_range(float4 (&acc)[CH], int beg, int end, int g, int gl, int lane,
                                             const int32_t* __restrict__ col, const float* __restrict__ sscale,
                                             const float4* __restrict__ x, int64_t ldx4, int nvec GCNSA_DBG_PARAM) {
  constexpr int NG = 32 / G;
  for (int base = beg; base < end; base += 32) {
    const int n = min(32, end - base);
    const int mine = lane < n ? __ldg(col + base + lane) : 0;
    const float msc = SCALED && lane < n ? __ldg(sscale + mine) : 1.f;
    for (int k0 = 0; k0 < n; k0 += NG * RU) {
      float4 v[RU][CH];
#pragma unroll
      for (int u = 0; u < RU; ++u) {
        const int k = k0 + u * NG + g;
        const int c = __shfl_sync(kFull, mine, k & 31);
        bool live = k < n;
#if GCNSA_DBG
        if (live && dbg.src_rows >= 0) live = dbg_in(&g_dbg_spmm, c, 0, dbg.src_rows, kDbgColumn);
#endif
        const float4* xr = x + (int64_t)c * ldx4 + gl;
#pragma unroll
        for (int ch = 0; ch < CH; ++ch)
          v[u][ch] = live && gl + ch * G < nvec ? __ldg(xr + ch * G) : make_float4(0.f, 0.f, 0.f, 0.f);
      }
#pragma unroll
      for (int u = 0; u < RU; ++u) {
        const float sc = SCALED ? __shfl_sync(kFull, msc, (k0 + u * NG + g) & 31) : 1.f;
#pragma unroll
        for (int ch = 0; ch < CH; ++ch) {
          if (SCALED) fma4(acc[ch], sc, v[u][ch]);
          else add4(acc[ch], v[u][ch]);
        }
      }
    }
  }
}

template <int G, int CH, int RU, bool SCALED>
__global__ void __launch_bounds__(256)
spmm_rest(int n_long, int n_rows, const int32_t* __restrict__ rowptr, const int32_t* __restrict__ rowend,
          const int32_t* __restrict__ col, const float* __restrict__ sscale, const float* __restrict__ rscale,
          const int32_t* __restrict__ order, const float4* __restrict__ x, int64_t ldx4, int nvec, int f, int epi,
          const float* __restrict__ aux, int64_t ldaux, float* __restrict__ y, int64_t ldy, const SpmmBase base GCNSA_DBG_PARAM) {
  wait_for_predecessors();
  constexpr int W = 8;
  __shared__ float4 part[W][G * CH];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, g = lane / G, gl = lane % G;
  const bool hub = (int)blockIdx.x < n_long;  // a hub row's entries are shared out to the warps of a block
  const int w = hub ? (int)blockIdx.x : n_long + ((int)blockIdx.x - n_long) * W + warp;
  if (w >= n_rows) return;
  const int row = order ? __ldg(order + w) : w;
  const bool whole = base.beyond && __ldcg(base.beyond) != 0;  // no partial sums: all entries of the row
#if GCNSA_DBG
  if (dbg.mat_rows >= 0 && !dbg_in(&g_dbg_spmm, row, 0, dbg.mat_rows, kDbgOrderEntry)) return;  // hub: whole block alike
#endif
  int beg = __ldg((whole ? base.all_rowptr : rowptr) + row), end = __ldg((whole ? base.all_rowptr + 1 : rowend) + row);
  if (whole) col = base.all_col;
#if GCNSA_DBG
  const int64_t nnz = whole ? base.all_nnz : dbg.nnz;
  if (!dbg_in(&g_dbg_spmm, beg, 0, (long long)end + 1, kDbgRowRange)) return;
  if (nnz >= 0 && !dbg_in(&g_dbg_spmm, end, 0, nnz + 1, kDbgRowRange)) return;
#endif
  float4 pieces[CH], acc[CH];
#pragma unroll
  for (int ch = 0; ch < CH; ++ch) pieces[ch] = acc[ch] = make_float4(0.f, 0.f, 0.f, 0.f);
  if (g == 0 && (!hub || warp == 0) && !whole) load_pieces<CH>(pieces, base, row, gl, G, nvec);
  if (hub) {
    const int share = (end - beg + W - 1) / W;
    beg = min(end, beg + warp * share);
    end = min(end, beg + share);
  }
  gather_range<G, CH, RU, SCALED>(acc, beg, end, g, gl, lane, col, sscale, x, ldx4, nvec GCNSA_DBG_ARG);
  fold_groups<G, CH>(acc);
  if (hub) {
    if (g == 0) {
#pragma unroll
      for (int ch = 0; ch < CH; ++ch) part[warp][gl + ch * G] = acc[ch];
    }
    __syncthreads();
    if (warp != 0) return;
  }
  if (g != 0) return;
  const float sc = rscale ? __ldg(rscale + row) : 1.f;
#pragma unroll
  for (int ch = 0; ch < CH; ++ch) {
    const int qq = gl + ch * G;
    if (qq >= nvec) continue;
    float4 r = acc[ch];
    if (hub) {
#pragma unroll
      for (int k = 1; k < W; ++k) add4(r, part[k][qq]);
    }
    add4(r, pieces[ch]);
    if (rscale) { r.x *= sc; r.y *= sc; r.z *= sc; r.w *= sc; }
    store_chunk(r, row, qq, f, epi, aux, ldaux, y, ldy);
  }
}

struct RestArgs {
  cudaStream_t s;
  int n_rows, n_long;
  const int32_t *rowptr, *rowend, *col, *order;
  const float *sscale, *rscale;
  int64_t ldx;
  int epi;
  int64_t ldaux, ldy;
  SpmmBounds dbg;
};
template <int G, int CH, int RU>
cudaError_t run_rest(const RestArgs& a, const float* x, int nvec, int f, const float* aux, float* y, const SpmmBase& base) {
  const int grid = a.n_long + (a.n_rows - a.n_long + 7) / 8;
  if (a.sscale)
    launch(spmm_rest<G, CH, RU, true>, grid, 256, 0, a.s, a.n_long, a.n_rows, a.rowptr, a.rowend, a.col, a.sscale, a.rscale, a.order,
                                                      reinterpret_cast<const float4*>(x), a.ldx / 4, nvec, f, a.epi, aux, a.ldaux,
                                                      y, a.ldy, base GCNSA_DBG_LAUNCH_ARG);
  else
    launch(spmm_rest<G, CH, RU, false>, grid, 256, 0, a.s, a.n_long, a.n_rows, a.rowptr, a.rowend, a.col, nullptr, a.rscale, a.order,
                                                       reinterpret_cast<const float4*>(x), a.ldx / 4, nvec, f, a.epi, aux,
                                                       a.ldaux, y, a.ldy, base GCNSA_DBG_LAUNCH_ARG);
  note_launch();
  return cudaGetLastError();
}

}  // namespace

int launch_spmm(void* stream, int64_t n_rows, const int32_t* rowptr, const int32_t* col, const float* val,
                const float* row_scale, const int32_t* order, int64_t n_long, const float* x, int64_t ldx, int32_t f, int32_t epi, const float* aux,
                int64_t ldaux, float* y, int64_t ldy, const SpmmBounds& bounds, const RowSplit& split) {
  if (n_rows == 0 || f == 0) return 0;
  Args a;
  a.dbg = bounds;
  a.s = (cudaStream_t)stream;
  a.n_rows = (int)n_rows;
  a.rowptr = rowptr; a.col = col; a.val = val; a.rscale = row_scale; a.order = order;
  a.n_long = order ? (int)std::min<int64_t>(std::max<int64_t>(n_long, 0), n_rows) : 0;
  a.n_warp = (int)n_rows;
  if (split.order) {
    a.order = split.order;
    a.n_long = (int)split.n_long;
    a.n_warp = (int)split.n_warp;
  }
  a.ldx = ldx; a.epi = epi; a.ldaux = ldaux; a.ldy = ldy;
  // 16-byte index loads need 16-byte aligned arrays; otherwise every quad goes element by element
  a.vec_idx = (((uintptr_t)col | (uintptr_t)val) & 15) == 0 ? 1 : 0;  // val == NULL (unit entries) counts as aligned
  const int nvec_total = (f + 3) / 4;
  // Column slabs of at most 5 x 32 float4 (640 floats) per launch.  Where the gathers have no locality, the gathered
  // matrix is larger than L2 and its rows cut to 128 bytes are not (each die of the chip keeps its own copy of what its
  // SMs read, so about 60 MB count), slabs of 8 float4 turn HBM reads into L2 hits: 400 000 rows of the degree-32 random
  // graph, F' = 256: 1 128 -> 829 us, 128: 530 -> 410, 64: 206 -> 192.  Where neighbouring rows share their columns the
  // slabs cost (245 000 rows of the 2.45 M-vertex graph, 256: 593 -> 764 us).
  constexpr int64_t kL2 = 96 << 20, kL2Shared = 60 << 20;
  const bool narrow = split.scattered && bounds.src_rows * nvec_total * 16 > kL2 && bounds.src_rows * 128 <= kL2Shared;
  const int step = narrow ? 8 : 160;
  for (int v0 = 0; v0 < nvec_total; v0 += step) {
    a.nvec = std::min(step, nvec_total - v0);
    a.x = x + 4 * v0;
    a.y = y + 4 * v0;
    a.aux = aux ? aux + 4 * v0 : nullptr;  // bias and mask are both indexed by column
    a.f = min(f - 4 * v0, 4 * a.nvec);
    cudaError_t e;
    const int nv = a.nvec;
    // MINB (blocks per SM the register allocation must allow) is part of the tuning: the kernel is bound by the
    // L1 data path, and about 32-40 resident warps per SM (64 resp. 48 registers a thread) measured fastest;
    // left alone the compiler unrolls to over 100 registers (16 warps), and at 32 registers (64 warps) L1 thrashes.
    if (nv <= 4) e = run<4, 1, 2, 128, 10, 4, 1, 8>(a);
    else if (nv <= 8) e = run<4, 2, 2, 128, 10, 8, 1, 8>(a);
    else if (nv <= 12) e = run<4, 3, 2, 128, 10, 16, 1, 8>(a);
    else if (nv <= 16) e = run<8, 2, 2, 128, 10, 16, 1, 8>(a);
    else if (nv <= 32) e = run<32, 1, 4, 256, 4, 32, 1, 8>(a);
    else if (nv <= 64) e = run<32, 2, 4, 256, 4, 32, 2, 4>(a);
    else if (nv <= 96) e = run<32, 3, 2, 256, 3, 32, 3, 2>(a);
    else if (nv <= 128) e = run<32, 4, 2, 256, 3, 32, 4, 2>(a);
    else e = run<32, 5, 2, 256, 3, 32, 5, 2>(a);
    if (e != cudaSuccess) return (int)e;
  }
  return 0;
}

int launch_spmm_rest(void* stream, int64_t n_rows, const int32_t* rowptr, const int32_t* rowend, const int32_t* col,
                     const float* row_scale, const float* src_scale, const int32_t* order, int64_t n_long, const float* x,
                     int64_t ldx, int32_t f, int32_t epi, const float* aux, int64_t ldaux, float* y, int64_t ldy,
                     const SpmmBase& base, const SpmmBounds& bounds) {
  if (n_rows == 0 || f == 0) return 0;
  RestArgs a;
  a.dbg = bounds;
  a.s = (cudaStream_t)stream;
  a.n_rows = (int)n_rows;
  a.n_long = order ? (int)std::min<int64_t>(std::max<int64_t>(n_long, 0), n_rows) : 0;
  a.rowptr = rowptr; a.rowend = rowend; a.col = col; a.order = order;
  a.sscale = src_scale; a.rscale = row_scale;
  a.ldx = ldx; a.epi = epi; a.ldaux = ldaux; a.ldy = ldy;
  const int nvec_total = (f + 3) / 4;
  for (int v0 = 0; v0 < nvec_total; v0 += 128) {  // column slabs of at most 4 x 32 float4
    SpmmBase b = base;
    b.q0 = v0;
    const int nv = std::min(128, nvec_total - v0), fs = std::min(f - 4 * v0, 4 * nv);
    const float* xs = x + 4 * v0;
    const float* as = aux ? aux + 4 * v0 : nullptr;
    float* ys = y + 4 * v0;
    cudaError_t e;
    if (nv <= 4) e = run_rest<4, 1, 2>(a, xs, nv, fs, as, ys, b);
    else if (nv <= 8) e = run_rest<8, 1, 4>(a, xs, nv, fs, as, ys, b);
    else if (nv <= 16) e = run_rest<16, 1, 4>(a, xs, nv, fs, as, ys, b);
    else if (nv <= 32) e = run_rest<32, 1, 8>(a, xs, nv, fs, as, ys, b);
    else if (nv <= 64) e = run_rest<32, 2, 4>(a, xs, nv, fs, as, ys, b);
    else e = run_rest<32, 4, 2>(a, xs, nv, fs, as, ys, b);
    if (e != cudaSuccess) return (int)e;
  }
  return 0;
}

int debug_word_spmm(unsigned long long* out, bool clear) {
  *out = 0ull;
#if GCNSA_DBG
  cudaError_t e = cudaMemcpyFromSymbol(out, g_dbg_spmm, sizeof(*out));
  if (e == cudaSuccess && clear) {
    const unsigned long long zero = 0ull;
    e = cudaMemcpyToSymbol(g_dbg_spmm, &zero, sizeof(zero));
  }
  return (int)e;
#else
  (void)clear;
  return 0;
#endif
}

}  // namespace gcnsa
