// GraphSAGE with the mean aggregator on the extended partitions (Section 4.1,
// "Investigated GCNs"; training scheme of Section 3.2): per mini-batch
//   1. a fixed number of neighbours is sampled for every vertex the batch needs
//      (the r smallest 64-bit selection keys among the vertex's neighbours
//      inside its extended partition: a uniform draw without replacement that
//      depends on (seed, partition, epoch, layer, vertex) only),
//   2. every layer is h_v = sigma([h_v | mean of the sampled neighbours] W + b),
//      the concatenation form of the published mean aggregator: the rows
//      [self | mean] are assembled by one gather kernel and multiplied by the
//      stacked matrix [W_self ; W_neigh] on the tensor cores,
//   3. softmax cross-entropy over the batch, the chain rule backwards (the mean
//      over a vertex's samples hands each sample 1 / count of the gradient),
//      one Adam step on the worker's copy of the parameters.
// The batch is laid out in slots: rows [0, nb) are the batch's vertices, row
// nb + i r2 + s is the s-th sampled neighbour of vertex i (r2 = fan-out of the
// output layer).  A vertex that several batch vertices sampled gets several
// slots; its embedding is the same in each (the hidden layer's sample depends
// on the vertex only), so the result is that of the definition and the
// backward pass needs no scatter: every slot has exactly one reader.
// All shapes are known to the host (batch size, fan-outs), so no step waits for
// a device value.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstring>
#include <new>
#include <string>
#include <vector>

#include "internal.h"
#include "launch.h"
#include "parts.h"

namespace gcnsa {

namespace {

constexpr unsigned kFull = 0xffffffffu;
typedef unsigned long long u64;

// SplitMix64 finalizer (Steele, Lea, Flood 2014) and the selection key built from it: the words are absorbed one
// at a time, the vertex id last
__host__ __device__ inline u64 mix64s(u64 z) {
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ULL;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBULL;
  return z ^ (z >> 31);
}
__host__ __device__ inline u64 key_prefix(u64 seed, u64 w0, u64 w1, u64 w2, u64 w3) {
  u64 h = mix64s(seed);
  h = mix64s(h ^ w0);
  h = mix64s(h ^ w1);
  h = mix64s(h ^ w2);
  return mix64s(h ^ w3);
}
constexpr u64 kTagNeighbor = 3, kTagBatch = 4;

inline unsigned blocks_for(int64_t items, int per_block) {
  return (unsigned)std::max<int64_t>(1, (items + per_block - 1) / per_block);
}

// ---------------------------------------------------------------- batches ---
// keys[i] = key(seed; 4, p, epoch, 0; list[i])
__global__ void sage_keys(const int32_t* __restrict__ list, int64_t n, u64 prefix, u64* __restrict__ keys) {
  wait_for_predecessors();
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) keys[i] = mix64s(prefix ^ (u64)list[i]);
}
// order[rank of keys[i]] = list[i]; keys are distinct (the key is a bijection of the vertex id), so the ranks are a
// permutation.  Brute force over tiles of keys in shared memory: n^2 comparisons, a millisecond at n = 10^5.
__global__ void __launch_bounds__(256)
sage_rank(const int32_t* __restrict__ list, const u64* __restrict__ keys, int64_t n, int32_t* __restrict__ order) {
  wait_for_predecessors();
  __shared__ u64 tile[1024];
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const u64 mine = i < n ? keys[i] : 0ull;
  int64_t rank = 0;
  for (int64_t t0 = 0; t0 < n; t0 += 1024) {
    const int cnt = (int)min((int64_t)1024, n - t0);
    for (int k = threadIdx.x; k < cnt; k += 256) tile[k] = keys[t0 + k];
    __syncthreads();
    if (i < n)
      for (int k = 0; k < cnt; ++k) rank += tile[k] < mine;
    __syncthreads();
  }
  if (i < n) order[rank] = list[i];
}

// --------------------------------------------------------------- sampling ---
// One warp per vertex vs[j] (-1 = none): its neighbours are the columns of its row of A + I other than itself.
// At most r of them: all, ascending.  More: the r with the smallest keys mix(prefix_v ^ u) (keys are distinct), in
// key order; out row j is padded with -1.
//
// Selection, r <= kFastR: one pipelined pass over the row collects the neighbours whose key is at most a threshold T
// into the warp's shared-memory list; the keys are uniform 64-bit numbers, so T = 2.5 r / deg of the key range
// catches about 2.5 r of them.  Between r and kCand candidates: their ranks among themselves (all pairs) are their
// ranks in the row, and ranks below r are the sample.  Fewer than r or more than kCand (rare): T is doubled / halved
// until both sides are bracketed, then bisected, and the pass repeated; the result never depends on T.
// Larger r: r rounds of "smallest key above the last one taken".
constexpr int kSampleWarps = 8, kCand = 128, kFastR = 50;

__global__ void __launch_bounds__(kSampleWarps * 32)
sage_sample(const int32_t* __restrict__ rowptr, const int32_t* __restrict__ col, const int32_t* __restrict__ vs,
            int64_t n_v, int r, u64 seed, u64 p, u64 epoch_layer, const int64_t* __restrict__ batch_state,
            int32_t* __restrict__ out, int32_t* __restrict__ cnt) {
  wait_for_predecessors();
  // recorded batches: the epoch is read from the batch state, epoch_layer then carries the layer only
  if (batch_state) epoch_layer += (u64)batch_state[1] * 256;
  __shared__ u64 cand_key[kSampleWarps][kCand];
  __shared__ int32_t cand_id[kSampleWarps][kCand];
  const int64_t j = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  if (j >= n_v) return;
  int32_t* row = out + j * r;
  const int v = vs[j];
  if (v < 0) {
    for (int s = lane; s < r; s += 32) row[s] = -1;
    if (lane == 0) cnt[j] = 0;
    return;
  }
  const int beg = rowptr[v], end = rowptr[v + 1];
  const int deg = end - beg - 1;  // the self-loop is stored exactly once
  if (deg <= r) {
    for (int e = beg + lane; e < end; e += 32) {
      const int u = col[e];
      if (u < v) row[e - beg] = u;
      else if (u > v) row[e - beg - 1] = u;
    }
    for (int s = max(deg, 0) + lane; s < r; s += 32) row[s] = -1;
    if (lane == 0) cnt[j] = max(deg, 0);
    return;
  }
  const u64 prefix = key_prefix(seed, kTagNeighbor, p, epoch_layer, (u64)v);
  if (r <= kFastR) {
    u64* ck = cand_key[wib];
    int32_t* ci = cand_id[wib];
    const double want = 2.5 * (double)r / (double)deg;
    u64 T = want >= 1.0 ? ~0ull : (u64)(want * 18446744073709551615.0);
    u64 lo = 0ull, hi = ~0ull;       // count(lo) < r (or nothing known), count(hi) > kCand (or nothing known)
    bool have_lo = false, have_hi = false;
    int n_c = 0;
    for (int attempt = 0; attempt < 200; ++attempt) {   // every retry shrinks [lo, hi]; 64 bisections always suffice
      n_c = 0;
      // eight loads a lane in flight while the eight before them are hashed: a hub row of thousands of neighbours is a
      // chain of load latencies, and the longest row of a batch sets the time of the kernel
      constexpr int kAhead = 8;
      int us[kAhead];
      auto load = [&](int e0) {
#pragma unroll
        for (int t = 0; t < kAhead; ++t) {
          const int e = e0 + 32 * t + lane;
          us[t] = e < end ? __ldg(col + e) : v;
        }
      };
      load(beg);
      for (int e0 = beg; e0 < end; e0 += 32 * kAhead) {
        int cur[kAhead];
#pragma unroll
        for (int t = 0; t < kAhead; ++t) cur[t] = us[t];
        if (e0 + 32 * kAhead < end) load(e0 + 32 * kAhead);
#pragma unroll
        for (int t = 0; t < kAhead; ++t) {
          if (e0 + 32 * t >= end) break;
          const int u = cur[t];
          const u64 k = mix64s(prefix ^ (u64)u);
          const bool take = u != v && k <= T;
          const unsigned m = __ballot_sync(kFull, take);
          if (take) {
            const int at = n_c + __popc(m & ((1u << lane) - 1));
            if (at < kCand) { ck[at] = k; ci[at] = u; }
          }
          n_c += __popc(m);
        }
      }
      if (n_c >= r && n_c <= kCand) break;
      if (n_c < r) { lo = T; have_lo = true; } else { hi = T; have_hi = true; }
      if (have_lo && have_hi) T = lo + (hi - lo) / 2;
      else if (have_lo) T = T > (~0ull >> 1) ? ~0ull : T * 2 + 1;
      else T = T / 2;
    }
    __syncwarp();
    for (int i = lane; i < n_c; i += 32) {
      const u64 mine = ck[i];
      int rank = 0;
      for (int q = 0; q < n_c; ++q) rank += ck[q] < mine;
      if (rank < r) row[rank] = ci[i];
    }
    if (lane == 0) cnt[j] = r;
    return;
  }
  u64 last = 0ull;
  for (int s = 0; s < r; ++s) {
    u64 best = 0ull;
    int who = -1;
    for (int e = beg + lane; e < end; e += 32) {
      const int u = col[e];
      if (u == v) continue;
      const u64 k = mix64s(prefix ^ (u64)u);
      if ((s == 0 || k > last) && (who < 0 || k < best)) { best = k; who = u; }
    }
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) {
      const u64 ob = __shfl_xor_sync(kFull, best, off);
      const int ow = __shfl_xor_sync(kFull, who, off);
      if (ow >= 0 && (who < 0 || ob < best)) { best = ob; who = ow; }
    }
    if (lane == 0) row[s] = who;
    last = best;
  }
  if (lane == 0) cnt[j] = r;
}

// ------------------------------------------------------ [self | mean] rows ---
// out[j] = [ src[self_j] | mean over the samples of row j of src[.] ], both halves ld floats wide (f of them
// meaningful, the rest zero).  self_idx == NULL: self_j = j.  samp == NULL: the samples of row j are the rows
// slot_base + j r + s, s < cnt[j] (the slot layout of the batch).  A row without a vertex (self_j < 0) is zero.
// A thread owns one float4 of one row and has eight of the samples' loads in flight (a warp per row with one sample after
// the other: 29.5 us a launch in the epoch of five workers side by side, this 16.2; 2 816 rows of 26 x 2 432 bytes).
__global__ void __launch_bounds__(256)
sage_concat_mean(const float* __restrict__ src, int64_t ld_src, int f, const int32_t* __restrict__ self_idx,
                 const int32_t* __restrict__ samp, const int32_t* __restrict__ cnt, int r, int64_t slot_base,
                 int64_t n_rows, float* __restrict__ out, int64_t ld) {
  wait_for_predecessors();
  const int lvec = (int)(ld / 4), nvec = (f + 3) / 4;
  const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= n_rows * lvec) return;
  const int64_t j = idx / lvec;
  const int q = (int)(idx - j * lvec);
  float4* o_self = reinterpret_cast<float4*>(out + j * 2 * ld);
  const int64_t self = self_idx ? (int64_t)__ldg(self_idx + j) : j;
  float4 a = make_float4(0.f, 0.f, 0.f, 0.f), m = a;
  if (q < nvec && self >= 0) {
    const int c = __ldg(cnt + j);
    const float4* col = reinterpret_cast<const float4*>(src) + q;
    const int64_t ld4 = ld_src / 4;
    a = __ldg(col + self * ld4);
#pragma unroll 8
    for (int s = 0; s < c; ++s) {
      const int64_t u = samp ? (int64_t)__ldg(samp + j * r + s) : slot_base + j * r + s;
      const float4 t = __ldg(col + u * ld4);
      m.x += t.x; m.y += t.y; m.z += t.z; m.w += t.w;
    }
    const float inv = c > 0 ? 1.0f / (float)c : 0.f;
    m.x *= inv; m.y *= inv; m.z *= inv; m.w *= inv;
  }
  o_self[q] = a;
  o_self[lvec + q] = m;
}

__global__ void sage_gather_labels(const int32_t* __restrict__ y, const int32_t* __restrict__ targets, int64_t nb,
                                   int32_t* __restrict__ yb) {
  wait_for_predecessors();
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < nb) yb[i] = y[targets[i]];
}

// Gradient w.r.t. the hidden layer's pre-activation, slot by slot.  dcat = G W^T has the layout of the [self | mean]
// rows: columns [0, ldh) belong to the batch vertex's own embedding, columns [ldh, 2 ldh) to the mean over its
// samples, of which each sample receives 1 / count.  ReLU'(z) = [h > 0].
__global__ void sage_hidden_grad(const float* __restrict__ dcat, const float* __restrict__ h1, const int32_t* __restrict__ cnt2,
                                 int64_t nb, int r2, int64_t ldh, int64_t n_rows, float* __restrict__ dz1) {
  wait_for_predecessors();
  const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= n_rows * ldh) return;
  const int64_t j = idx / ldh, c = idx - j * ldh;
  float g = 0.f;
  if (j < nb) {
    g = dcat[j * 2 * ldh + c];
  } else {
    const int64_t i = (j - nb) / r2, s = (j - nb) - i * r2;
    const int k = cnt2[i];
    if (s < k) g = dcat[i * 2 * ldh + ldh + c] / (float)k;
  }
  dz1[idx] = h1[idx] > 0.f ? g : 0.f;
}

// The output layer of a batch and everything that a batch vertex's slots need from it, in one kernel: [h_v | mean h_u] W2 + b2,
// softmax cross-entropy, the gradient dcat = g W2^T of the [self | mean] row and, sample by sample, the gradient of the hidden
// layer's pre-activation.  A slot has one reader, so a block that holds kHeadRows vertices needs nothing of the others: what
// was a chain of launches (gather, labels, product, softmax, product, gradient, column sums) is one, in fp32 FMAs.
// What bounds it is latency: a few thousand FMAs a thread's worth of work, W2 (at most kHeadWeights floats) from L2 by every
// block, so the loads of a phase are independent of one another and spread over all 256 threads.
// Partial sums for the loss and both bias gradients leave one row per block, added up in block order by a later launch.
// 20 000 vertices in batches of 256 (hidden 128, 20 classes): 2 330 -> 2 120 us per epoch; 116 483 (41 classes): 19.7 -> 19.1 ms.
// Wider output layers and larger batches stay on the tensor cores: their products are work, not latency.  Epochs of workers side by
// side, one kernel against the launches: 64 to 256 x 20 to 64 in batches of 64 take 0.73 to 0.79 of the time, of 256 0.79 to 0.99; with
// batches of 1 024 128 x 20 0.92, 128 x 47 0.97, 128 x 64 1.09, 64 x 256 1.36; with 4 096 128 x 20 1.03, 64 x 256 1.57.  Up to 16 classes take
// 0.82 to 1.02 in batches of 4 096.  So the lines are batch x classes (logits, softmax) and batch x weights (both products).
constexpr int kHeadRows = 2, kHeadThreads = 256;
constexpr int64_t kHeadWeights = 32768, kHeadBatch = 4096, kHeadFewClasses = 16, kHeadBatchClasses = 45000, kHeadBatchWeights = 12 << 20;
bool head_pays(int64_t batch, int64_t ldh, int64_t ldc, int64_t c) {
  if (batch > kHeadBatch || c > 256 || ldh > 1024 || 2 * ldh * ldc > kHeadWeights) return false;
  return c <= kHeadFewClasses || (batch * c <= kHeadBatchClasses && batch * 2 * ldh * ldc <= kHeadBatchWeights);
}
struct Head {
  const float* h1;
  int ldh;
  const int32_t* cnt2;
  int r2, nb;
  const float* w2;
  int ldc, c, qp;  // qp: lanes per k in the forward product, a power of two and at least the quads of c
  const float* b2;
  const int32_t *y, *vertices;  // the label of row i is y[vertices[i]]
  float inv_nb;
  float *cat2, *logits, *g, *dz1;
  float *loss_part, *g_sums, *dz_sums;  // [blocks], [blocks x 4 quads], [blocks x ldh]
};
__global__ void __launch_bounds__(kHeadThreads) sage_head(const Head p) {
  wait_for_predecessors();
  constexpr int V = kHeadRows, T = kHeadThreads;
  extern __shared__ float4 head_smem[];
  __shared__ float sh_loss[V];
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const int K = 2 * p.ldh, lv = p.ldh / 4, quads = (p.c + 3) / 4, cp = 4 * p.qp, v0 = blockIdx.x * V;
  float* cat = reinterpret_cast<float*>(head_smem);  // [V][K]
  float* dcat = cat + V * K;                         // [V][K]
  float* part = dcat + V * K;                        // [slices][V][cp]; later [row lanes][ldh]
  float* gs = part + 4 * T * V;                      // [V][cp]
  for (int i = t; i < V * lv; i += T) {
    const int v = i / lv, q = i - v * lv, row = v0 + v;
    float4 a = make_float4(0.f, 0.f, 0.f, 0.f), m = a;
    if (row < p.nb) {
      const int n = __ldg(p.cnt2 + row);
      const float4* col = reinterpret_cast<const float4*>(p.h1) + q;
      a = __ldg(col + (int64_t)row * lv);
      const float4* samp = col + ((int64_t)p.nb + (int64_t)row * p.r2) * lv;
#pragma unroll 8
      for (int s = 0; s < n; ++s) {
        const float4 x = __ldg(samp + (int64_t)s * lv);
        m.x += x.x; m.y += x.y; m.z += x.z; m.w += x.w;
      }
      const float inv = n > 0 ? 1.0f / (float)n : 0.f;
      m.x *= inv; m.y *= inv; m.z *= inv; m.w *= inv;
      float4* out = reinterpret_cast<float4*>(p.cat2 + (int64_t)row * K);  // the weight gradient's product reads it
      out[q] = a;
      out[lv + q] = m;
    }
    reinterpret_cast<float4*>(cat + v * K)[q] = a;
    reinterpret_cast<float4*>(cat + v * K)[lv + q] = m;
  }
  __syncthreads();
  {  // logits: thread = four classes of a slice of k
    const int q = t & (p.qp - 1), slice = t / p.qp, slices = T / p.qp, per = (K + slices - 1) / slices;
    const int k0 = slice * per, k1 = min(K, k0 + per);
    float4 acc[V];
#pragma unroll
    for (int v = 0; v < V; ++v) acc[v] = make_float4(0.f, 0.f, 0.f, 0.f);
    if (q < quads) {
#pragma unroll 8
      for (int k = k0; k < k1; ++k) {
        const float4 w = __ldg(reinterpret_cast<const float4*>(p.w2 + (int64_t)k * p.ldc) + q);
#pragma unroll
        for (int v = 0; v < V; ++v) {
          const float x = cat[v * K + k];
          acc[v].x = fmaf(x, w.x, acc[v].x); acc[v].y = fmaf(x, w.y, acc[v].y);
          acc[v].z = fmaf(x, w.z, acc[v].z); acc[v].w = fmaf(x, w.w, acc[v].w);
        }
      }
    }
#pragma unroll
    for (int v = 0; v < V; ++v) reinterpret_cast<float4*>(part + (slice * V + v) * cp)[q] = acc[v];
  }
  __syncthreads();
  if (warp < V) {  // softmax: a warp per vertex, up to 256 classes
    const int v = warp, row = v0 + v, slices = T / p.qp;
    const bool in = row < p.nb;
    const int yi = in ? __ldg(p.y + __ldg(p.vertices + row)) : 0;
    float z[8], mx = -INFINITY, zy = -INFINITY;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int j = lane + 32 * i;
      z[i] = -INFINITY;
      if (j < p.c) {
        float sum = 0.f;
        for (int k = 0; k < slices; ++k) sum += part[(k * V + v) * cp + j];
        z[i] = sum + __ldg(p.b2 + j);
        if (in) p.logits[(int64_t)row * p.ldc + j] = z[i];
        if (j == yi) zy = z[i];
      }
      mx = fmaxf(mx, z[i]);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(kFull, mx, o));
    zy = __shfl_sync(kFull, zy, yi & 31);
    float se = 0.f;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      z[i] = expf(z[i] - mx);
      if (lane + 32 * i < p.c) se += z[i];
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) se += __shfl_xor_sync(kFull, se, o);
    const float inv_se = 1.f / se;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int j = lane + 32 * i;
      if (j >= 4 * quads) continue;
      const float d = in && j < p.c ? (z[i] * inv_se - (j == yi ? 1.f : 0.f)) * p.inv_nb : 0.f;
      gs[v * cp + j] = d;
      if (in) p.g[(int64_t)row * p.ldc + j] = d;
    }
    if (lane == 0) sh_loss[v] = in ? (mx + logf(se)) - zy : 0.f;
  }
  __syncthreads();
  if (t == 0) {
    float sum = 0.f;
#pragma unroll
    for (int v = 0; v < V; ++v) sum += sh_loss[v];
    p.loss_part[blockIdx.x] = sum;
  }
  for (int j = t; j < 4 * quads; j += T) {
    float sum = 0.f;
#pragma unroll
    for (int v = 0; v < V; ++v) sum += gs[v * cp + j];
    p.g_sums[(int64_t)blockIdx.x * 4 * quads + j] = sum;
  }
  for (int k = t; k < K; k += T) {  // dcat = g W2^T (W2's lines are in L1 by now)
    const float4* w = reinterpret_cast<const float4*>(p.w2 + (int64_t)k * p.ldc);
    float sum[V];
#pragma unroll
    for (int v = 0; v < V; ++v) sum[v] = 0.f;
#pragma unroll 4
    for (int q = 0; q < quads; ++q) {
      const float4 x = __ldg(w + q);
#pragma unroll
      for (int v = 0; v < V; ++v) {
        const float4 d = reinterpret_cast<const float4*>(gs + v * cp)[q];
        sum[v] = fmaf(d.x, x.x, fmaf(d.y, x.y, fmaf(d.z, x.z, fmaf(d.w, x.w, sum[v]))));
      }
    }
#pragma unroll
    for (int v = 0; v < V; ++v) dcat[v * K + k] = sum[v];
  }
  __syncthreads();
  // hidden gradient, ReLU'(z) = [h > 0]: the vertex's own slot takes the first half of dcat, each of its samples 1 / count of the
  // second; thread = four features of every ny-th slot
  const int q = t % lv, ry = t / lv, ny = T / lv, slots = 1 + p.r2;
  float4 sum = make_float4(0.f, 0.f, 0.f, 0.f);
  if (ry < ny) {
#pragma unroll 4
    for (int i = ry; i < V * slots; i += ny) {
      const int v = i / slots, s = i - v * slots - 1, row = v0 + v;  // s = -1: the vertex itself
      if (row >= p.nb) break;
      const int64_t slot = s < 0 ? row : p.nb + (int64_t)row * p.r2 + s;
      const float4 h = __ldg(reinterpret_cast<const float4*>(p.h1) + slot * lv + q);
      float4 d = make_float4(0.f, 0.f, 0.f, 0.f);
      if (s < 0) {
        d = reinterpret_cast<const float4*>(dcat + v * K)[q];
      } else {
        const int n = __ldg(p.cnt2 + row);
        if (s < n) {
          d = reinterpret_cast<const float4*>(dcat + v * K)[lv + q];
          const float den = (float)n;
          d.x /= den; d.y /= den; d.z /= den; d.w /= den;
        }
      }
      d.x = h.x > 0.f ? d.x : 0.f; d.y = h.y > 0.f ? d.y : 0.f; d.z = h.z > 0.f ? d.z : 0.f; d.w = h.w > 0.f ? d.w : 0.f;
      reinterpret_cast<float4*>(p.dz1)[slot * lv + q] = d;
      sum.x += d.x; sum.y += d.y; sum.z += d.z; sum.w += d.w;
    }
    reinterpret_cast<float4*>(part)[ry * lv + q] = sum;
  }
  __syncthreads();
  for (int i = t; i < lv; i += T) {
    float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int k = 0; k < ny; ++k) {
      const float4 b = reinterpret_cast<const float4*>(part)[k * lv + i];
      a.x += b.x; a.y += b.y; a.z += b.z; a.w += b.w;
    }
    reinterpret_cast<float4*>(p.dz_sums)[(int64_t)blockIdx.x * lv + i] = a;
  }
}
// loss[0] = mean of the batch's losses from the blocks' partial sums (in block order by lane), loss[1] += their sum
__global__ void sage_head_loss(const float* __restrict__ part, int count, float inv_nb, float weight, float* loss) {
  wait_for_predecessors();
  float s = 0.f;
  for (int i = threadIdx.x; i < count; i += 32) s += part[i];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(kFull, s, o);
  if (threadIdx.x == 0) {
    loss[0] = s * inv_nb;
    loss[1] += loss[0] * weight;
  }
}

// out[0] += number of source rows the [self | mean] kernel reads for these rows: 1 + cnt per row that has a vertex
__global__ void sage_count_reads(const int32_t* __restrict__ self_idx, const int32_t* __restrict__ cnt, int64_t n_rows,
                                 u64* out) {
  wait_for_predecessors();
  const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  int c = 0;
  if (j < n_rows && (!self_idx || self_idx[j] >= 0)) c = 1 + cnt[j];
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) c += __shfl_xor_sync(kFull, c, off);
  if ((threadIdx.x & 31) == 0 && c) atomicAdd(out, (u64)c);
}

// acc[0] += loss * weight (one thread): the running sum of the batch losses of a partition
// Batch state of the recorded batches: [0] = index of the batch in flight, [1] = epoch.  A replayed graph cannot
// take new kernel arguments, so the batch's first kernel advances the index itself and copies the batch's targets.
__global__ void sage_set_state(int64_t* state, int64_t b, int64_t epoch) {
  wait_for_predecessors();
  state[0] = b;
  state[1] = epoch;
}
// one block: every thread reads the old index before thread 0 writes the new one
__global__ void sage_begin_batch(int64_t* state, const int32_t* __restrict__ order, int batch, int32_t* __restrict__ targets) {
  wait_for_predecessors();
  const int64_t b = state[0] + 1;
  __syncthreads();
  for (int i = threadIdx.x; i < batch; i += blockDim.x) targets[i] = order[b * batch + i];
  if (threadIdx.x == 0) state[0] = b;
}

__global__ void sage_loss_add(float* acc, const float* loss, float weight) {
  wait_for_predecessors();
  if (threadIdx.x == 0 && blockIdx.x == 0) acc[0] += loss[0] * weight;
}
// dst[0] = part[0] * scale; part[0] = 0: a worker's epoch is over
__global__ void sage_loss_fold(float* dst, float* part, float scale) {
  wait_for_predecessors();
  if (threadIdx.x == 0 && blockIdx.x == 0) {
    dst[0] = part[0] * scale;
    part[0] = 0.f;
  }
}
// The end of an epoch (Section 3.2): theta = mean of the workers' copies [m x count], added in worker order; the
// working copy of the last worker becomes theta as well; loss[0] = sum of the workers' losses.
__global__ void sage_param_mean(int64_t count, int m, const float* copies, float* __restrict__ theta, float* work,
                                float scale, const float* __restrict__ loss_parts,
                                float* __restrict__ loss) {
  wait_for_predecessors();
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < count) {
    float acc = 0.f;
    for (int p = 0; p < m; ++p) acc = fmaf(copies[(int64_t)p * count + i], scale, acc);
    theta[i] = acc;
    work[i] = acc;
  }
  if (i == 0) {
    float sum = 0.f;
    for (int p = 0; p < m; ++p) sum += loss_parts[p];
    loss[0] = sum;
  }
}

}  // namespace
}  // namespace gcnsa

using namespace gcnsa;

// Everything one worker's batches need: order, samples, activations, gradient, scratch.  An epoch runs several
// workers at once, one per lane.
struct SageLane {
  float* grad = nullptr;
  // batch order of one (partition, epoch)
  u64* keys = nullptr;
  int32_t* order = nullptr;
  int32_t order_p = -1;
  int64_t order_epoch = -1;
  uint64_t order_uid = 0;
  // the batch
  int32_t *b1 = nullptr, *cnt2 = nullptr, *s1 = nullptr, *cnt1 = nullptr, *yb = nullptr;
  float *cat1 = nullptr, *h1 = nullptr, *cat2 = nullptr, *logits = nullptr, *g = nullptr, *dcat2 = nullptr, *dz1 = nullptr, *ce_sums = nullptr;
  float *loss_part = nullptr, *g_sums = nullptr, *dz_sums = nullptr;  // of sage_head's blocks
  float* loss = nullptr;  // [0] batch loss, [1] sum over the worker's batches
  int64_t* batch_state = nullptr;
  void *ws = nullptr, *sc = nullptr;
};

struct gcnsa_sage {
  Env env;
  gcnsa_sage_opts o{};
  int32_t m = 0;
  int64_t f = 0, h = 0, c = 0, ldf = 0, ldh = 0, ldc = 0;
  int64_t count = 0, w1_off = 0, b1_off = 0, w2_off = 0, b2_off = 0;  // flat parameter layout
  int64_t max_rows1 = 0;  // batch (1 + r2): rows of the hidden layer per batch
  int64_t nt_max = 1;     // training vertices of the partition that has most
  int64_t epoch = 0;
  int head_qp = 0;        // 0: the output layer runs launch by launch; otherwise sage_head takes it (Head::qp)
  size_t head_smem = 0;
  // parameters: aggregated; per worker its copy and its moments ([m x count] each)
  float *theta = nullptr, *copies = nullptr, *am = nullptr, *av = nullptr;
  double* adam_state = nullptr;  // [m x 4]
  float* loss_parts = nullptr;   // [m] a worker's share of the epoch loss
  float* loss = nullptr;         // epoch loss
  uint8_t* ones = nullptr;
  size_t ws_bytes = 0;
  int beside = 1;  // workers an epoch may run at once
  std::vector<SageLane> lanes;   // lane 0 also serves the calls that go batch by batch
  std::vector<cudaStream_t> side;  // streams of lanes 1, 2, ...
  cudaEvent_t fork_ev = nullptr;
  std::vector<cudaEvent_t> join_ev;
  int work_p = 0;                // whose copy GCNSA_SAGE_WORK_* and the step-by-step calls address
  int64_t last_nb = 0, last_rows1 = 0;  // the latest batch, in the buffers of lane last_lane
  int last_lane = 0;
  // recorded full-size batch of every worker (batch_graph): keyed by the partitions object
  std::vector<cudaGraphExec_t> batch_exec;
  std::vector<int> batch_kernels;
  uint64_t batch_uid = 0;
  bool graph_off = false;
  // optional timing with CUDA events: classes 0 = [self | mean] gathers, 1 = dense products, 2 = everything else
  struct Rec { int cat; double bytes, flops; int64_t launches; };
  bool prof_on = false;
  std::vector<cudaEvent_t> ev;
  std::vector<Rec> recs;
  int64_t launches_mark = 0;
  u64* read_rows = nullptr;  // device: [0] source rows read by the hidden layer's gathers, [1] by the output layer's
  void prof_begin() {
    if (!prof_on) return;
    const size_t i = recs.size() * 2;
    while (ev.size() < i + 2) {
      cudaEvent_t e;
      if (cudaEventCreate(&e) != cudaSuccess) { prof_on = false; return; }
      ev.push_back(e);
    }
    launches_mark = gcnsa_launch_count();
    cudaEventRecord(ev[i], env.stream());
  }
  void prof_end(int cat, double bytes, double flops) {
    if (!prof_on) return;
    cudaEventRecord(ev[recs.size() * 2 + 1], env.stream());
    recs.push_back({cat, bytes, flops, gcnsa_launch_count() - launches_mark});
  }
  std::vector<void*> owned;
  void* dalloc(size_t bytes) {
    void* p = env.alloc(bytes);
    if (p) owned.push_back(p);
    return p;
  }
};

namespace {

int cuda_err(cudaError_t e, const char* what) { return fail(GCNSA_ERR_CUDA, std::string(what) + ": " + cudaGetErrorString(e)); }
#define SCK(call)                                        \
  do {                                                   \
    cudaError_t e_ = (call);                             \
    if (e_ != cudaSuccess) return cuda_err(e_, #call);   \
  } while (0)
#define SCKL(call)                                               \
  do {                                                           \
    int e_ = (call);                                             \
    if (e_ != 0) return cuda_err((cudaError_t)e_, #call);        \
  } while (0)
#define SLAUNCHED(what)                                          \
  do {                                                           \
    note_launch();                                               \
    cudaError_t e_ = cudaGetLastError();                         \
    if (e_ != cudaSuccess) return cuda_err(e_, what);            \
  } while (0)

int check_model(const gcnsa_sage* S, const gcnsa_parts* P) {
  if (!S || !P) return fail(GCNSA_ERR_ARG, "NULL argument");
  bool fits = P->m == S->m && P->f == S->f && P->c == S->c;
  for (const DevPart& d : P->parts) fits = fits && d.info.n_train <= S->nt_max;  // the batch order of a partition
  if (!fits) return fail(GCNSA_ERR_ARG, "model was created for other partitions");
  return GCNSA_OK;
}

// the batch order of (p, epoch): the loss-carrying vertices of the partition in ascending key order
int ensure_order(gcnsa_sage* S, const gcnsa_parts* P, int32_t p, int64_t epoch, SageLane& W, cudaStream_t s) {
  if (W.order_p == p && W.order_epoch == epoch && W.order_uid == P->uid) return GCNSA_OK;
  const DevPart& d = P->parts[p];
  const int64_t nt = d.info.n_train;
  if (nt > 0) {
    const u64 prefix = key_prefix(S->o.seed, kTagBatch, (u64)p, (u64)epoch, 0);
    launch(sage_keys, blocks_for(nt, 256), 256, 0, s, d.m_order, nt, prefix, W.keys);
    SLAUNCHED("sage_keys");
    launch(sage_rank, blocks_for(nt, 256), 256, 0, s, d.m_order, W.keys, nt, W.order);
    SLAUNCHED("sage_rank");
  }
  W.order_p = p; W.order_epoch = epoch; W.order_uid = P->uid;
  return GCNSA_OK;
}

int64_t n_batches(const gcnsa_sage* S, const gcnsa_parts* P, int32_t p) {
  return (P->parts[p].info.n_train + S->o.batch - 1) / S->o.batch;
}

// recorded = true: the launches are being captured for replay; the batch index and the epoch then come from
// W.batch_state on the device (a full-size batch), b and epoch are not used
int run_batch(gcnsa_sage* S, const gcnsa_parts* P, int32_t p, int64_t epoch, int64_t b, bool apply, SageLane& W, cudaStream_t s,
              bool recorded = false) {
  int rc = recorded ? GCNSA_OK : ensure_order(S, P, p, epoch, W, s);
  if (rc) return rc;
  const DevPart& d = P->parts[p];
  void* sv = s;
  const int64_t nt = d.info.n_train, B = S->o.batch;
  const int64_t nb = recorded ? B : std::min<int64_t>(B, nt - b * B);
  const int r1 = S->o.fanout[0], r2 = S->o.fanout[1];
  const int64_t rows1 = nb * (1 + r2);
  const int32_t* targets = W.order + b * B;
  const int mode = S->o.gemm_mode;

  // ---- the batch's vertices and their samples
  S->prof_begin();
  const int64_t* state = recorded ? W.batch_state : nullptr;
  const u64 ep = recorded ? 0 : (u64)epoch * 256;
  if (recorded) {
    launch(sage_begin_batch, 1, 256, 0, s, W.batch_state, W.order, (int)B, W.b1);
    SLAUNCHED("sage_begin_batch");
  } else {
    SCK(cudaMemcpyAsync(W.b1, targets, (size_t)nb * sizeof(int32_t), cudaMemcpyDeviceToDevice, s));
  }
  if (r2 > 0) {
    launch(sage_sample, blocks_for(nb * 32, kSampleWarps * 32), kSampleWarps * 32, 0, s, d.rowptr, d.col, W.b1, nb, r2, S->o.seed, (u64)p,
                                                        ep + 2, state, W.b1 + nb, W.cnt2);
    SLAUNCHED("sage_sample");
  } else {
    SCK(cudaMemsetAsync(W.cnt2, 0, (size_t)nb * sizeof(int32_t), s));
  }
  if (r1 > 0) {
    launch(sage_sample, blocks_for(rows1 * 32, kSampleWarps * 32), kSampleWarps * 32, 0, s, d.rowptr, d.col, W.b1, rows1, r1, S->o.seed, (u64)p,
                                                           ep + 1, state, W.s1, W.cnt1);
    SLAUNCHED("sage_sample");
  } else {
    SCK(cudaMemsetAsync(W.cnt1, 0, (size_t)rows1 * sizeof(int32_t), s));
  }
  if (S->prof_on) {
    launch(sage_count_reads, blocks_for(rows1, 256), 256, 0, s, W.b1, W.cnt1, rows1, S->read_rows);
    SLAUNCHED("sage_count_reads");
    launch(sage_count_reads, blocks_for(nb, 256), 256, 0, s, nullptr, W.cnt2, nb, S->read_rows + 1);
    SLAUNCHED("sage_count_reads");
  }
  S->prof_end(2, 0.0, 0.0);
  // ---- hidden layer: H1 = relu([x_v | mean x_u] [W_self ; W_neigh] + b)
  S->prof_begin();
  launch(sage_concat_mean, blocks_for(rows1 * (S->ldf / 4), 256), 256, 0, s, d.x, P->ldx, (int)S->f, W.b1, W.s1, W.cnt1, r1, 0, rows1,
                                                              W.cat1, S->ldf);
  SLAUNCHED("sage_concat_mean");
  S->prof_end(0, 8.0 * (double)rows1 * (double)S->ldf, 0.0);  // the rows written; the rows read are counted on the device
  float* w = S->copies + (size_t)p * S->count;
  const double fl1 = 2.0 * (double)rows1 * (double)S->h * 2.0 * (double)S->f, fl2 = 2.0 * (double)nb * (double)S->c * 2.0 * (double)S->h;
  S->prof_begin();
  SCKL(launch_gemm(sv, mode, 0, 0, rows1, S->h, 2 * S->ldf, W.cat1, 2 * S->ldf, w + S->w1_off, S->ldh, W.h1, S->ldh, 0,
                   GCNSA_EPI_BIAS_RELU, w + S->b1_off, 0, W.ws, S->ws_bytes, S->beside));
  S->prof_end(1, 0.0, fl1);
  float* gr = W.grad;
  if (S->head_qp > 0) {  // ---- output layer, loss and the gradient down to the hidden layer's pre-activation
    Head hd;
    hd.h1 = W.h1; hd.ldh = (int)S->ldh;
    hd.cnt2 = W.cnt2; hd.r2 = r2; hd.nb = (int)nb;
    hd.w2 = w + S->w2_off; hd.ldc = (int)S->ldc; hd.c = (int)S->c; hd.qp = S->head_qp;
    hd.b2 = w + S->b2_off; hd.y = d.y; hd.vertices = W.b1;
    hd.inv_nb = 1.0f / (float)nb;
    hd.cat2 = W.cat2; hd.logits = W.logits; hd.g = W.g; hd.dz1 = W.dz1;
    hd.loss_part = W.loss_part; hd.g_sums = W.g_sums; hd.dz_sums = W.dz_sums;
    const unsigned blocks = blocks_for(nb, kHeadRows);
    S->prof_begin();
    launch(sage_head, blocks, kHeadThreads, S->head_smem, s, hd);
    SLAUNCHED("sage_head");
    launch(sage_head_loss, 1, 32, 0, s, W.loss_part, (int)blocks, hd.inv_nb, (float)nb, W.loss);
    SLAUNCHED("sage_head_loss");
    SCKL(launch_sum_rows(sv, blocks, (int32_t)S->c, W.g_sums, (S->c + 3) / 4 * 4, gr + S->b2_off, 0, W.sc));
    SCKL(launch_sum_rows(sv, blocks, (int32_t)S->h, W.dz_sums, S->ldh, gr + S->b1_off, 0, W.sc));
    S->prof_end(2, 0.0, 2.0 * fl2);
    S->prof_begin();
    SCKL(launch_gemm(sv, mode, 1, 0, 2 * S->ldh, S->c, nb, W.cat2, 2 * S->ldh, W.g, S->ldc, gr + S->w2_off, S->ldc, 0,
                     GCNSA_EPI_NONE, nullptr, 0, W.ws, S->ws_bytes, S->beside));
    S->prof_end(1, 0.0, fl2);
  } else {
    // ---- output layer: logits = [h_v | mean h_u] [W_self ; W_neigh] + b, the samples of vertex i in slots nb + i r2 + s
    S->prof_begin();
    launch(sage_concat_mean, blocks_for(nb * (S->ldh / 4), 256), 256, 0, s, W.h1, S->ldh, (int)S->h, nullptr, nullptr, W.cnt2, r2, nb, nb,
                                                             W.cat2, S->ldh);
    SLAUNCHED("sage_concat_mean");
    S->prof_end(0, 8.0 * (double)nb * (double)S->ldh, 0.0);
    S->prof_begin();
    SCKL(launch_gemm(sv, mode, 0, 0, nb, S->c, 2 * S->ldh, W.cat2, 2 * S->ldh, w + S->w2_off, S->ldc, W.logits, S->ldc, 0,
                     GCNSA_EPI_BIAS, w + S->b2_off, 0, W.ws, S->ws_bytes, S->beside));
    S->prof_end(1, 0.0, fl2);
    // ---- loss over the batch and its gradient
    S->prof_begin();
    launch(sage_gather_labels, blocks_for(nb, 256), 256, 0, s, d.y, W.b1, nb, W.yb);
    SLAUNCHED("sage_gather_labels");
    CeSide side;  // the partial column sums of the logit gradient come with it
    if (ce_by_groups((int32_t)S->c)) side.sums = W.ce_sums;
    SCKL(launch_softmax_ce(sv, nb, (int32_t)S->c, W.logits, S->ldc, W.yb, S->ones, nb, W.loss, W.g, S->ldc, W.sc, side));
    launch(sage_loss_add, 1, 32, 0, s, W.loss + 1, W.loss, (float)nb);
    SLAUNCHED("sage_loss_add");
    S->prof_end(2, 0.0, 0.0);
    // ---- backward
    S->prof_begin();
    SCKL(launch_gemm(sv, mode, 1, 0, 2 * S->ldh, S->c, nb, W.cat2, 2 * S->ldh, W.g, S->ldc, gr + S->w2_off, S->ldc, 0,
                     GCNSA_EPI_NONE, nullptr, 0, W.ws, S->ws_bytes, S->beside));
    SCKL(launch_gemm(sv, mode, 0, 1, nb, 2 * S->ldh, S->c, W.g, S->ldc, w + S->w2_off, S->ldc, W.dcat2, 2 * S->ldh, 0,
                     GCNSA_EPI_NONE, nullptr, 0, W.ws, S->ws_bytes, S->beside));
    S->prof_end(1, 0.0, 2.0 * fl2);
    S->prof_begin();
    if (side.sums) {
      SCKL(launch_ce_sums(sv, nb, (int32_t)S->c, W.ce_sums, gr + S->b2_off, 0));
    } else {
      SCKL(launch_colsum(sv, nb, (int32_t)S->c, W.g, S->ldc, gr + S->b2_off, 0, W.sc));
    }
    launch(sage_hidden_grad, blocks_for(rows1 * S->ldh, 256), 256, 0, s, W.dcat2, W.h1, W.cnt2, nb, std::max(r2, 1), S->ldh, rows1,
                                                                    W.dz1);
    SLAUNCHED("sage_hidden_grad");
    S->prof_end(2, 0.0, 0.0);
  }
  S->prof_begin();
  SCKL(launch_gemm(sv, mode, 1, 0, 2 * S->ldf, S->h, rows1, W.cat1, 2 * S->ldf, W.dz1, S->ldh, gr + S->w1_off, S->ldh, 0,
                   GCNSA_EPI_NONE, nullptr, 0, W.ws, S->ws_bytes, S->beside));
  S->prof_end(1, 0.0, fl1);
  S->prof_begin();
  if (S->head_qp == 0) SCKL(launch_colsum(sv, rows1, (int32_t)S->h, W.dz1, S->ldh, gr + S->b1_off, 0, W.sc));
  // ---- the worker's Adam step (its own moments and step count)
  if (apply) {
    double* st = S->adam_state + 4 * (size_t)p;
    SCKL(launch_adam_advance(sv, st, S->o.beta1, S->o.beta2));
    SCKL(launch_adam_dev(sv, S->count, w, W.grad, S->am + (size_t)p * S->count, S->av + (size_t)p * S->count, 1.0f,
                         S->o.lr, S->o.beta1, S->o.beta2, S->o.eps, st));
  }
  S->prof_end(2, 0.0, 0.0);
  S->last_nb = nb;
  S->last_rows1 = rows1;
  return GCNSA_OK;
}

}  // namespace

extern "C" {

int gcnsa_sage_destroy(gcnsa_sage* S) {
  if (!S) return GCNSA_OK;
  cudaStreamSynchronize(S->env.stream());
  for (cudaStream_t st : S->side) cudaStreamSynchronize(st);
  for (void* p : S->owned) S->env.release(p);
  for (cudaEvent_t e : S->ev) cudaEventDestroy(e);
  for (cudaGraphExec_t g : S->batch_exec)
    if (g) cudaGraphExecDestroy(g);
  for (cudaStream_t st : S->side) cudaStreamDestroy(st);
  for (cudaEvent_t e : S->join_ev) cudaEventDestroy(e);
  if (S->fork_ev) cudaEventDestroy(S->fork_ev);
  delete S;
  return GCNSA_OK;
}

// How many workers an epoch runs at once: up to eight while a batch has at most kLaneRows rows in the hidden layer.  The
// kernels of a batch (13, or two dozen) are a chain of microseconds on a fraction of the SMs, so workers side by side overlap
// (116 K vertices, 5 workers, batches of 256: 63.2 ms per epoch with one lane, 47.7 with two, 38.4 with four, 29.9
// with five; 20 000 vertices, 4 workers: 7.7 -> 4.2 ms).  Larger batches fill the chip by themselves and their lanes
// would cost gigabytes.  The lanes after the first take at most 1 GB (a batch of 2 816 rows of 602 features 17 MB each; with
// fan-outs in the thousands the sample lists alone can be half a gigabyte).  The default stream runs one worker at a time.
constexpr int64_t kLaneRows = 32768;
static int sage_lanes(int32_t m, int64_t max_rows1, size_t lane_bytes, cudaStream_t s) {
  constexpr size_t kLaneBytes = (size_t)1 << 30;
  if (max_rows1 > kLaneRows || s == nullptr) return 1;
  return (int)std::min<int64_t>(std::min<int>(m, 8), 1 + (int64_t)(kLaneBytes / lane_bytes));
}

int gcnsa_sage_create(const gcnsa_env* env, const gcnsa_parts* parts, const gcnsa_sage_opts* opts,
                      const float* const* w_self0, const float* const* w_neigh0, const float* const* b0, gcnsa_sage** out) {
  if (!out) return fail(GCNSA_ERR_ARG, "out is NULL");
  *out = nullptr;
  if (!env || !parts || !opts || !w_self0 || !w_neigh0) return fail(GCNSA_ERR_ARG, "NULL argument");
  if (opts->dims[0] != parts->f || opts->dims[2] != parts->c || opts->dims[1] < 1)
    return fail(GCNSA_ERR_ARG, "dims[0] must equal f, dims[2] must equal c of the partitions, dims[1] >= 1");
  if (opts->fanout[0] < 0 || opts->fanout[1] < 0 || opts->fanout[0] > 4096 || opts->fanout[1] > 4096 || opts->batch < 1 ||
      opts->batch > 65536)
    return fail(GCNSA_ERR_ARG, "fan-outs must be in [0, 4096] and the batch size in [1, 65536]");
  if (opts->gemm_mode != GCNSA_GEMM_FP32 && opts->gemm_mode != GCNSA_GEMM_TF32X3 && opts->gemm_mode != GCNSA_GEMM_TF32) return fail(GCNSA_ERR_ARG, "unknown gemm_mode");
  if (!(opts->lr > 0.f) || !(opts->beta1 >= 0.f && opts->beta1 < 1.f) || !(opts->beta2 >= 0.f && opts->beta2 < 1.f) ||
      !(opts->eps > 0.f))
    return fail(GCNSA_ERR_ARG, "Adam hyper-parameters out of range");
  for (int l = 0; l < 2; ++l)
    if (!w_self0[l] || !w_neigh0[l]) return fail(GCNSA_ERR_ARG, "w_self0[l] or w_neigh0[l] is NULL");
  int dev_count = 0;
  if (cudaGetDeviceCount(&dev_count) != cudaSuccess || dev_count == 0) {
    cudaGetLastError();
    return fail(GCNSA_ERR_CUDA, "no CUDA device: this library has no CPU fallback");
  }
  gcnsa_sage* S = new (std::nothrow) gcnsa_sage();
  if (!S) return fail(GCNSA_ERR_OOM, "host allocation failed");
  S->env.e = *env;
  S->o = *opts;
  S->m = parts->m;
  S->f = opts->dims[0]; S->h = opts->dims[1]; S->c = opts->dims[2];
  S->ldf = GCNSA_LD(S->f); S->ldh = GCNSA_LD(S->h); S->ldc = GCNSA_LD(S->c);
  auto up64 = [](int64_t v) { return (v + 63) / 64 * 64; };
  int64_t off = 0;
  S->w1_off = off; off += up64(2 * S->ldf * S->ldh);
  S->b1_off = off; off += up64(S->ldh);
  S->w2_off = off; off += up64(2 * S->ldh * S->ldc);
  S->b2_off = off; off += up64(S->ldc);
  S->count = off;
  const int64_t B = opts->batch, r1 = opts->fanout[0], r2 = opts->fanout[1];
  S->max_rows1 = B * (1 + r2);
  for (const DevPart& d : parts->parts) S->nt_max = std::max<int64_t>(S->nt_max, d.info.n_train);
  auto fail_free = [&](int code) {
    const std::string keep = gcnsa_last_error();
    gcnsa_sage_destroy(S);
    return fail(code, keep);
  };
  const size_t pb = (size_t)S->count * sizeof(float);
  struct Want { void** slot; size_t bytes; };
  size_t ws = 0;
  const int mode = opts->gemm_mode;
  ws = std::max(ws, gemm_workspace(mode, 0, 0, S->max_rows1, S->h, 2 * S->ldf));
  ws = std::max(ws, gemm_workspace(mode, 0, 0, B, S->c, 2 * S->ldh));
  ws = std::max(ws, gemm_workspace(mode, 1, 0, 2 * S->ldh, S->c, B));
  ws = std::max(ws, gemm_workspace(mode, 0, 1, B, 2 * S->ldh, S->c));
  ws = std::max(ws, gemm_workspace(mode, 1, 0, 2 * S->ldf, S->h, S->max_rows1));
  // the last batch of a partition is smaller: its products have their own split along the inner dimension
  for (int64_t nb = 1; nb < B; ++nb) {
    ws = std::max(ws, gemm_workspace(mode, 0, 0, nb * (1 + r2), S->h, 2 * S->ldf));
    ws = std::max(ws, gemm_workspace(mode, 1, 0, 2 * S->ldf, S->h, nb * (1 + r2)));
    ws = std::max(ws, gemm_workspace(mode, 1, 0, 2 * S->ldh, S->c, nb));
    ws = std::max(ws, gemm_workspace(mode, 0, 1, nb, 2 * S->ldh, S->c));
    ws = std::max(ws, gemm_workspace(mode, 0, 0, nb, S->c, 2 * S->ldh));
  }
  S->ws_bytes = ws;
  const size_t sc = std::max(std::max(softmax_ce_scratch(B), colsum_scratch(S->max_rows1, (int32_t)S->h)),
                             colsum_scratch(B, (int32_t)S->c));
  // Small output layers (the 41 classes of a 128-wide hidden layer: 12 288 floats of W2) are one kernel; plain TF32 keeps its
  // products on the tensor cores, which is what that mode is there to measure.
  if (mode != GCNSA_GEMM_TF32 && head_pays(B, S->ldh, S->ldc, S->c)) {
    S->head_qp = 1;
    while (4 * S->head_qp < S->c) S->head_qp *= 2;
    S->head_smem = sizeof(float) * (size_t)(kHeadRows * (4 * S->ldh + 4 * kHeadThreads + 4 * S->head_qp));
  }
  const size_t head_blocks = S->head_qp ? blocks_for(B, kHeadRows) : 0;
  const size_t f4 = sizeof(float), i4 = sizeof(int32_t);
  std::vector<Want> wants = {{(void**)&S->theta, pb}, {(void**)&S->copies, pb * (size_t)S->m},
                             {(void**)&S->am, pb * (size_t)S->m}, {(void**)&S->av, pb * (size_t)S->m},
                             {(void**)&S->adam_state, sizeof(double) * 4 * (size_t)S->m},
                             {(void**)&S->loss_parts, f4 * (size_t)S->m}, {(void**)&S->loss, f4},
                             {(void**)&S->ones, (size_t)B}, {(void**)&S->read_rows, sizeof(u64) * 2}};
  auto lane_wants = [&](SageLane& W) {
    return std::vector<Want>{
        {(void**)&W.grad, pb}, {(void**)&W.keys, sizeof(u64) * (size_t)S->nt_max}, {(void**)&W.order, i4 * (size_t)S->nt_max},
        {(void**)&W.b1, i4 * (size_t)S->max_rows1}, {(void**)&W.cnt2, i4 * (size_t)B},
        {(void**)&W.s1, i4 * (size_t)(S->max_rows1 * std::max<int64_t>(r1, 1))},
        {(void**)&W.cnt1, i4 * (size_t)S->max_rows1}, {(void**)&W.yb, i4 * (size_t)B},
        {(void**)&W.cat1, f4 * (size_t)(S->max_rows1 * 2 * S->ldf)}, {(void**)&W.h1, f4 * (size_t)(S->max_rows1 * S->ldh)},
        {(void**)&W.cat2, f4 * (size_t)(B * 2 * S->ldh)}, {(void**)&W.logits, f4 * (size_t)(B * S->ldc)},
        {(void**)&W.g, f4 * (size_t)(B * S->ldc)}, {(void**)&W.dcat2, f4 * (size_t)(B * 2 * S->ldh)},
        {(void**)&W.dz1, f4 * (size_t)(S->max_rows1 * S->ldh)}, {(void**)&W.ce_sums, ce_sums_scratch((int32_t)S->c)}, {(void**)&W.loss, f4 * 2},
        {(void**)&W.loss_part, f4 * head_blocks}, {(void**)&W.g_sums, f4 * head_blocks * (size_t)((S->c + 3) / 4 * 4)},
        {(void**)&W.dz_sums, f4 * head_blocks * (size_t)S->ldh},
        {(void**)&W.batch_state, sizeof(int64_t) * 2}, {&W.ws, ws}, {&W.sc, std::max<size_t>(sc, 256)}};
  };
  cudaStream_t s = S->env.stream();
  auto obtain = [&](const std::vector<Want>& list) {
    for (const Want& w : list) {
      *w.slot = S->dalloc(std::max<size_t>(w.bytes, 256));
      if (!*w.slot) return fail(GCNSA_ERR_OOM, "device allocation failed");
      const cudaError_t e = cudaMemsetAsync(*w.slot, 0, std::max<size_t>(w.bytes, 256), s);
      if (e != cudaSuccess) return cuda_err(e, "cudaMemsetAsync");
    }
    return (int)GCNSA_OK;
  };
  int rc = obtain(wants);
  S->lanes.resize(1);
  size_t lane_bytes = 0;
  for (const Want& w : lane_wants(S->lanes[0])) lane_bytes += std::max<size_t>(w.bytes, 256);
  S->lanes.resize((size_t)sage_lanes(S->m, S->max_rows1, lane_bytes, s));
  if (S->max_rows1 <= kLaneRows) S->beside = std::min(S->m, 3);
  for (size_t i = 0; i < S->lanes.size() && rc == GCNSA_OK; ++i) {
    const size_t mark = S->owned.size();
    rc = obtain(lane_wants(S->lanes[i]));
    if (rc == GCNSA_ERR_OOM && i > 0) {  // lanes after the first only make the epoch faster
      while (S->owned.size() > mark) {
        S->env.release(S->owned.back());
        S->owned.pop_back();
      }
      S->lanes.resize(i);
      rc = GCNSA_OK;
      break;
    }
  }
  if (rc != GCNSA_OK) return fail_free(rc);
  cudaError_t e = cudaEventCreateWithFlags(&S->fork_ev, cudaEventDisableTiming);
  for (size_t i = 1; i < S->lanes.size() && e == cudaSuccess; ++i) {
    cudaStream_t st;
    cudaEvent_t ev;
    e = cudaStreamCreateWithFlags(&st, cudaStreamNonBlocking);
    if (e == cudaSuccess) {
      S->side.push_back(st);
      e = cudaEventCreateWithFlags(&ev, cudaEventDisableTiming);
      if (e == cudaSuccess) S->join_ev.push_back(ev);
    }
  }
  if (e == cudaSuccess) e = cudaMemsetAsync(S->ones, 1, (size_t)B, s);
  // initial parameters: W_self in rows [0, f) of the stacked matrix, W_neigh in rows [ld, ld + f)
  const int64_t din[2] = {S->f, S->h}, dout[2] = {S->h, S->c}, ldin[2] = {S->ldf, S->ldh}, ldo[2] = {S->ldh, S->ldc};
  const int64_t w_off[2] = {S->w1_off, S->w2_off}, b_off[2] = {S->b1_off, S->b2_off};
  for (int l = 0; l < 2 && e == cudaSuccess; ++l) {
    float* wd = S->theta + w_off[l];
    const size_t hp = (size_t)dout[l] * sizeof(float), dp = (size_t)ldo[l] * sizeof(float);
    e = cudaMemcpy2DAsync(wd, dp, w_self0[l], hp, hp, (size_t)din[l], cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess)
      e = cudaMemcpy2DAsync(wd + ldin[l] * ldo[l], dp, w_neigh0[l], hp, hp, (size_t)din[l], cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess && b0 && b0[l])
      e = cudaMemcpyAsync(S->theta + b_off[l], b0[l], hp, cudaMemcpyHostToDevice, s);
  }
  for (int32_t p = 0; p < S->m && e == cudaSuccess; ++p)
    e = cudaMemcpyAsync(S->copies + (size_t)p * S->count, S->theta, pb, cudaMemcpyDeviceToDevice, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) {
    cuda_err(e, "upload of the initial parameters");
    return fail_free(GCNSA_ERR_CUDA);
  }
  *out = S;
  return GCNSA_OK;
}

int gcnsa_sage_batches(const gcnsa_sage* S, const gcnsa_parts* P, int32_t p, int64_t* count_out) {
  int rc = check_model(S, P);
  if (rc) return rc;
  if (!count_out || p < 0 || p >= P->m) return fail(GCNSA_ERR_ARG, "bad partition index or NULL");
  *count_out = n_batches(S, P, p);
  return GCNSA_OK;
}

int gcnsa_sage_batch(gcnsa_sage* S, const gcnsa_parts* P, int32_t p, int64_t epoch, int64_t b, int32_t apply,
                     float* loss_dev) {
  int rc = check_model(S, P);
  if (rc) return rc;
  if (p < 0 || p >= P->m || epoch < 0 || epoch >= (1LL << 40)) return fail(GCNSA_ERR_ARG, "partition index or epoch out of range");
  if (b < 0 || b >= n_batches(S, P, p)) return fail(GCNSA_ERR_ARG, "batch index out of range");
  // the working copy as it stands: the one of the worker that ran last
  cudaStream_t s = S->env.stream();
  if (S->work_p != p)
    SCK(cudaMemcpyAsync(S->copies + (size_t)p * S->count, S->copies + (size_t)S->work_p * S->count,
                        (size_t)S->count * sizeof(float), cudaMemcpyDeviceToDevice, s));
  S->work_p = p;
  S->last_lane = 0;
  SageLane& W = S->lanes[0];
  rc = run_batch(S, P, p, epoch, b, apply != 0, W, s);
  if (rc) return rc;
  if (loss_dev) SCK(cudaMemcpyAsync(loss_dev, W.loss, sizeof(float), cudaMemcpyDeviceToDevice, s));
  return GCNSA_OK;
}

// the graph of worker p's full-size batch in lane W, recorded on stream s unless it is there already
static int ensure_batch_graph(gcnsa_sage* S, const gcnsa_parts* P, int32_t p, SageLane& W, cudaStream_t s) {
  if (S->batch_uid != P->uid || (int32_t)S->batch_exec.size() != P->m) {
    for (cudaGraphExec_t g : S->batch_exec)
      if (g) cudaGraphExecDestroy(g);
    S->batch_exec.assign((size_t)P->m, nullptr);
    S->batch_kernels.assign((size_t)P->m, 0);
    S->batch_uid = P->uid;
  }
  if (S->batch_exec[p]) return GCNSA_OK;
  const int64_t launches0 = gcnsa_launch_count();
  cudaGraph_t graph = nullptr;
  if (cudaStreamBeginCapture(s, cudaStreamCaptureModeThreadLocal) == cudaSuccess) {
    const int rc = run_batch(S, P, p, S->epoch, 0, true, W, s, true);
    const cudaError_t e = cudaStreamEndCapture(s, &graph);
    const int recorded = (int)(gcnsa_launch_count() - launches0);
    note_launch(-recorded);  // recorded, not launched
    if (rc != GCNSA_OK || e != cudaSuccess || !graph || cudaGraphInstantiate(&S->batch_exec[p], graph, 0) != cudaSuccess) {
      S->batch_exec[p] = nullptr;
      S->graph_off = true;  // this stream or driver cannot record a batch: plain launches from now on
    }
    S->batch_kernels[p] = recorded;
    if (graph) cudaGraphDestroy(graph);
    cudaGetLastError();
  } else {
    cudaGetLastError();
    S->graph_off = true;
  }
  return GCNSA_OK;
}

int gcnsa_sage_epoch(gcnsa_sage* S, const gcnsa_parts* P, float* loss_dev) {
  int rc = check_model(S, P);
  if (rc) return rc;
  cudaStream_t s = S->env.stream();
  const size_t pb = (size_t)S->count * sizeof(float);
  // Workers are independent within an epoch: lane i takes workers ..., counted from the last one backwards in steps of
  // the number of lanes (lane 0 ends with the last worker), each lane on a stream of its own.
  const int lanes = S->prof_on || s == nullptr ? 1 : (int)S->lanes.size();
  auto stream_of = [&](int lane) { return lane == 0 ? s : S->side[lane - 1]; };
  if (lanes > 1) {
    SCK(cudaEventRecord(S->fork_ev, s));
    for (int i = 1; i < lanes; ++i) SCK(cudaStreamWaitEvent(stream_of(i), S->fork_ev, 0));
  }
  // where a lane stands: worker p, its next batch, its batches and how many of them are replayed
  struct At { int32_t p; int64_t b, nbatch, nreplay; };
  std::vector<At> at((size_t)lanes);
  auto begin = [&](int lane, int32_t p) -> int {
    SageLane& W = S->lanes[lane];
    cudaStream_t st = stream_of(lane);
    At& a = at[lane];
    a.p = p; a.b = 0; a.nbatch = n_batches(S, P, p); a.nreplay = 0;
    // the worker starts the epoch from the aggregated parameters (Section 3.2)
    SCK(cudaMemcpyAsync(S->copies + (size_t)p * S->count, S->theta, pb, cudaMemcpyDeviceToDevice, st));
    SCK(cudaMemsetAsync(W.loss + 1, 0, sizeof(float), st));
    // the worker's full-size batches are one kernel sequence with the same shapes: recorded once per worker and
    // replayed, the batch index advancing on the device; the ragged last batch runs as plain launches
    const int64_t nfull = P->parts[p].info.n_train / S->o.batch;
    if (S->o.batch_graph && !S->graph_off && !S->prof_on && s != nullptr && nfull > 1) {
      int r = ensure_order(S, P, p, S->epoch, W, st);
      if (r == GCNSA_OK) r = ensure_batch_graph(S, P, p, W, st);
      if (r) return r;
      if (S->batch_exec[p]) {
        launch(sage_set_state, 1, 1, 0, st, W.batch_state, -1, S->epoch);
        SLAUNCHED("sage_set_state");
        a.nreplay = nfull;
      }
    }
    return GCNSA_OK;
  };
  auto finish = [&](int lane) -> int {
    const int32_t p = at[lane].p;
    const int64_t nt = P->parts[p].info.n_train;
    launch(sage_loss_fold, 1, 32, 0, stream_of(lane), S->loss_parts + p, S->lanes[lane].loss + 1,
                                                  nt > 0 ? 1.0f / ((float)nt * (float)P->m) : 0.f);
    SLAUNCHED("sage_loss_fold");
    return GCNSA_OK;
  };
  auto workers = [&]() -> int {
    int open = 0;
    for (int i = 0; i < lanes; ++i) {
      const int32_t first = (P->m - 1 - i) % lanes;  // the smallest p with (m - 1 - p) % lanes == i
      const int r = begin(i, first);
      if (r) return r;
      ++open;
    }
    while (open > 0) {  // one batch of every lane in turn, so that all streams are fed
      for (int i = 0; i < lanes; ++i) {
        At& a = at[i];
        if (a.p < 0) continue;
        if (a.b < a.nreplay) {
          SCK(cudaGraphLaunch(S->batch_exec[a.p], stream_of(i)));
          note_launch(S->batch_kernels[a.p]);
          S->last_nb = S->o.batch;
          S->last_rows1 = (int64_t)S->o.batch * (1 + S->o.fanout[1]);
          ++a.b;
        } else if (a.b < a.nbatch) {
          const int r = run_batch(S, P, a.p, S->epoch, a.b, true, S->lanes[i], stream_of(i));
          if (r) return r;
          ++a.b;
        }
        if (a.b < a.nbatch) continue;
        int r = finish(i);
        if (r) return r;
        const int32_t next = a.p + lanes;
        if (next < P->m) {
          r = begin(i, next);
          if (r) return r;
        } else {
          a.p = -1;
          --open;
        }
      }
    }
    return GCNSA_OK;
  };
  rc = workers();
  // (also when a worker has failed: what the others have been given ends before what follows on the caller's stream)
  for (int i = 1; i < lanes; ++i) {
    SCK(cudaEventRecord(S->join_ev[i - 1], stream_of(i)));
    SCK(cudaStreamWaitEvent(s, S->join_ev[i - 1], 0));
  }
  if (rc) return rc;
  // what gcnsa_sage_batch_export describes: the last batch of the last worker that has any
  for (int32_t p = P->m - 1; p >= 0; --p) {
    const int64_t nt = P->parts[p].info.n_train;
    if (nt == 0) continue;
    S->last_nb = nt - (n_batches(S, P, p) - 1) * S->o.batch;
    S->last_rows1 = S->last_nb * (1 + S->o.fanout[1]);
    S->last_lane = (P->m - 1 - p) % lanes;
    break;
  }
  S->work_p = P->m - 1;
  launch(sage_param_mean, blocks_for(S->count, 256), 256, 0, s, S->count, P->m, S->copies, S->theta,
                                                            S->copies + (size_t)S->work_p * S->count, 1.0f / (float)P->m,
                                                            S->loss_parts, S->loss);
  SLAUNCHED("sage_param_mean");
  if (loss_dev) SCK(cudaMemcpyAsync(loss_dev, S->loss, sizeof(float), cudaMemcpyDeviceToDevice, s));
  S->epoch += 1;
  return GCNSA_OK;
}

int gcnsa_sage_profile(gcnsa_sage* S, int32_t enable) {
  if (!S) return fail(GCNSA_ERR_ARG, "model is NULL");
  SCK(cudaStreamSynchronize(S->env.stream()));
  S->prof_on = enable != 0;
  S->recs.clear();
  SCK(cudaMemsetAsync(S->read_rows, 0, 2 * sizeof(u64), S->env.stream()));
  return GCNSA_OK;
}

int gcnsa_sage_profile_read(gcnsa_sage* S, gcnsa_profile* out) {
  if (!S || !out) return fail(GCNSA_ERR_ARG, "NULL argument");
  std::memset(out, 0, sizeof(*out));
  SCK(cudaStreamSynchronize(S->env.stream()));
  for (size_t i = 0; i < S->recs.size(); ++i) {
    float ms = 0.f;
    SCK(cudaEventElapsedTime(&ms, S->ev[2 * i], S->ev[2 * i + 1]));
    const auto& r = S->recs[i];
    out->ms[r.cat] += ms;
    out->launches[r.cat] += r.launches;
    out->alg_bytes[r.cat] += r.bytes;
    out->flops[r.cat] += r.flops;
  }
  u64 rows[2] = {0, 0};
  SCK(cudaMemcpy(rows, S->read_rows, sizeof(rows), cudaMemcpyDeviceToHost));
  out->alg_bytes[0] += 4.0 * (double)rows[0] * (double)S->f;
  out->alg_bytes[S->head_qp > 0 ? 2 : 0] += 4.0 * (double)rows[1] * (double)S->h;  // (sage_head gathers them itself)
  for (int c = 0; c < 3; ++c) { out->l1_bytes[c] = out->alg_bytes[c]; out->alg_bytes_val[c] = out->alg_bytes[c]; }
  S->recs.clear();
  SCK(cudaMemsetAsync(S->read_rows, 0, 2 * sizeof(u64), S->env.stream()));
  return GCNSA_OK;
}

int gcnsa_sage_get_epoch(const gcnsa_sage* S, int64_t* epoch_out) {
  if (!S || !epoch_out) return fail(GCNSA_ERR_ARG, "NULL argument");
  *epoch_out = S->epoch;
  return GCNSA_OK;
}

int gcnsa_sage_batch_shape(const gcnsa_sage* S, int64_t* nb_out, int64_t* rows1_out) {
  if (!S || !nb_out || !rows1_out) return fail(GCNSA_ERR_ARG, "NULL argument");
  *nb_out = S->last_nb;
  *rows1_out = S->last_rows1;
  return GCNSA_OK;
}

int gcnsa_sage_batch_export(const gcnsa_sage* S, const gcnsa_sage_batch_host* dst) {
  if (!S || !dst) return fail(GCNSA_ERR_ARG, "NULL argument");
  cudaStream_t s = S->env.stream();
  const size_t nb = (size_t)S->last_nb, rows1 = (size_t)S->last_rows1;
  const size_t r1 = (size_t)S->o.fanout[0];
  const SageLane& W = S->lanes[S->last_lane];
  if (dst->vertices && rows1) SCK(cudaMemcpyAsync(dst->vertices, W.b1, rows1 * sizeof(int32_t), cudaMemcpyDeviceToHost, s));
  if (dst->count2 && nb) SCK(cudaMemcpyAsync(dst->count2, W.cnt2, nb * sizeof(int32_t), cudaMemcpyDeviceToHost, s));
  if (dst->samples1 && rows1 && r1)
    SCK(cudaMemcpyAsync(dst->samples1, W.s1, rows1 * r1 * sizeof(int32_t), cudaMemcpyDeviceToHost, s));
  if (dst->count1 && rows1) SCK(cudaMemcpyAsync(dst->count1, W.cnt1, rows1 * sizeof(int32_t), cudaMemcpyDeviceToHost, s));
  if (dst->hidden && rows1)
    SCK(cudaMemcpy2DAsync(dst->hidden, (size_t)S->h * sizeof(float), W.h1, (size_t)S->ldh * sizeof(float),
                          (size_t)S->h * sizeof(float), rows1, cudaMemcpyDeviceToHost, s));
  if (dst->logits && nb)
    SCK(cudaMemcpy2DAsync(dst->logits, (size_t)S->c * sizeof(float), W.logits, (size_t)S->ldc * sizeof(float),
                          (size_t)S->c * sizeof(float), nb, cudaMemcpyDeviceToHost, s));
  if (dst->dlogits && nb)
    SCK(cudaMemcpy2DAsync(dst->dlogits, (size_t)S->c * sizeof(float), W.g, (size_t)S->ldc * sizeof(float),
                          (size_t)S->c * sizeof(float), nb, cudaMemcpyDeviceToHost, s));
  if (dst->loss) SCK(cudaMemcpyAsync(dst->loss, W.loss, sizeof(float), cudaMemcpyDeviceToHost, s));
  SCK(cudaStreamSynchronize(s));
  return GCNSA_OK;
}

static int sage_param(const gcnsa_sage* S, int32_t what, int32_t layer, float** base_out, int64_t* rows, int64_t* cols,
                      int64_t* ld) {
  if (!S) return fail(GCNSA_ERR_ARG, "model is NULL");
  if (layer < 0 || layer > 1) return fail(GCNSA_ERR_ARG, "layer out of range");
  const int kind = what % 3, which = what / 3;  // kind: self, neighbour, bias; which: aggregated, working copy, gradient
  float* buf = which == 0 ? S->theta : which == 1 ? S->copies + (size_t)S->work_p * S->count
                          : which == 2 ? S->lanes[S->last_lane].grad : nullptr;
  if (!buf || what < 0) return fail(GCNSA_ERR_ARG, "unknown tensor id");
  const int64_t din = layer == 0 ? S->f : S->h, dout = layer == 0 ? S->h : S->c;
  const int64_t ldin = layer == 0 ? S->ldf : S->ldh, ldo = layer == 0 ? S->ldh : S->ldc;
  const int64_t w_off = layer == 0 ? S->w1_off : S->w2_off, b_off = layer == 0 ? S->b1_off : S->b2_off;
  *cols = dout; *ld = ldo;
  if (kind == 2) { *base_out = buf + b_off; *rows = 1; }
  else { *base_out = buf + w_off + (kind == 1 ? ldin * ldo : 0); *rows = din; }
  return GCNSA_OK;
}

int gcnsa_sage_get(const gcnsa_sage* S, int32_t what, int32_t layer, void* host_dst, size_t bytes) {
  float* base = nullptr;
  int64_t rows = 0, cols = 0, ld = 0;
  int rc = sage_param(S, what, layer, &base, &rows, &cols, &ld);
  if (rc) return rc;
  if (!host_dst || bytes != (size_t)(rows * cols) * sizeof(float)) return fail(GCNSA_ERR_ARG, "NULL or byte count does not match");
  SCK(cudaMemcpy2DAsync(host_dst, (size_t)cols * sizeof(float), base, (size_t)ld * sizeof(float), (size_t)cols * sizeof(float),
                        (size_t)rows, cudaMemcpyDeviceToHost, S->env.stream()));
  SCK(cudaStreamSynchronize(S->env.stream()));
  return GCNSA_OK;
}

}  // extern "C"
