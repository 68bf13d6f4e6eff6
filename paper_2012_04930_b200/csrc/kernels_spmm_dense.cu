// The dense part of Y = B X, B the 0/1 pattern of A + I (Section 4.1 with the normalization factored out), on the
// tensor cores.
//
// In a graph whose vertex ids follow its communities a tile of 256 rows meets most of its columns many times (98 % of
// the entries of a 51 249-row partition of the 233 K-vertex graph lie in columns that at least four of the tile's rows
// share).  A warp per row gathers the source row once per entry; here a tile's shared columns are one contraction
// [256 x K] [K x F] whose left operand is a bit matrix.  Its entries are exact in bf16, and a fp32 source value is the
// exact sum of three bf16 terms (its 24 significant bits cut into 8 + 8 + 8), so three bf16 products per entry keep
// fp32 inputs; the accumulators are fp32.  The columns a tile shares too rarely stay in a remainder CSR that spmm_rest
// adds.
//
// split_rows cuts X into the three terms once; a source row of a slab of N <= 64 features is then one to three lines
// of 128 bytes, which cp.async puts where the MN-major, 128-byte swizzled tile of the MMA wants them.  (TMA's
// tile::gather4 fetches the same lines without a thread's help, but only four every 33 clocks: 1 600 clocks per unit.)
// A work unit is a chunk of 64 columns of one tile for one slab: 24 MMAs of 128 x N x 16, 768 clocks of the tensor pipe
// at N = 64.  The units of all tiles are one list that is cut into equal runs, one per CTA (one CTA per SM): a tile's
// run boundaries leave two partial sums, which spmm_rest adds in order.
//
// Roles: warps 0 and 7 issue the MMAs of the upper and the lower 128 rows (an issuing thread is held up until the tensor
// pipe takes its instruction, so while one of them waits for its operands the other keeps the pipe busy); warps 1-6
// fetch the source rows, every sixth unit each; warps 8-15 turn the bits of a row (thread = row) into bf16 words in
// tensor memory, the A operand; warps 16-23 fold finished accumulators into registers.
//
// The accumulator of the tensor core truncates when it adds: over the thousands of steps of a tile a bias of about
// 1e-8 per step would pass the rounding of an fp32 sum.  So an accumulator only lives for one unit and is then added to
// the thread's running sums with a rounded fp32 add, while the MMAs work in a second accumulator.
//
// A bit that is not set is a 0 that multiplies the source row, a set one a 2, and the split subtracts: with Inf or NaN in
// a source row all rows of the tiles that list its column would be NaN, and sums above half of the largest fp32 would
// overflow.  split_rows looks for such values (not finite, or 2^96 and more: below that twice the sum of 2^31 terms is
// finite) and leaves a word for spmm_rest, which then takes all entries of every row as gathers and no partial sums.
#include <cuda_runtime.h>

#include <algorithm>
#include <mutex>

#include "debug_check.h"
#include "internal.h"
#include "launch.h"
#include "tc_device.h"

namespace gcnsa {

namespace {

#if GCNSA_DBG
GCNSA_DBG_WORD(g_dbg_dense);
#endif

constexpr int kLoadWarp0 = 1, kLoadWarps = 6, kExpandWarp0 = 8, kFoldWarp0 = 16, kRowWarps = 8;
constexpr int kThreads = 32 * (kFoldWarp0 + kRowWarps);
constexpr int kStagesA = 4;           // chunks whose A is in tensor memory
constexpr int kStagesB = 8;           // chunks whose source rows are in (or on their way to) shared memory
// registers per thread by role, in multiples of 8; their sum over the six warpgroups is what the launch gives (80 each)
constexpr int kRegsLoad = 72, kRegsExpand = 48, kRegsFold = 120;
static_assert(2 * (kRegsLoad + kRegsExpand + kRegsFold) <= 6 * 80, "setmaxnreg draws on the registers of the launch");
constexpr int kLineBytes = 8 * 1024;  // 64 columns x 128 bytes: 8 groups of 8 columns
constexpr int kBitBytes = 2 * 1024;   // 256 rows x 64 bits

// How the three terms of a slab's features lie in a row's lines of 64 bf16: term t starts at feature t * STEP.
template <int N>
struct Lines {
  static constexpr int STEP = N <= 32 ? N : 64;
  static constexpr int COUNT = (3 * STEP + 63) / 64;
  static constexpr int STAGE = COUNT * kLineBytes + kBitBytes;  // ... and the bits of the chunk
  static constexpr int BAR_OFF = kStagesB * STAGE;
  // more than half of an SM's shared memory, so that two CTAs never share an SM (each takes all of tensor memory)
  static constexpr int SMEM = (BAR_OFF + 512 + 1024) > 118 * 1024 ? BAR_OFF + 512 + 1024 : 118 * 1024;
  static __host__ __device__ constexpr int offset(int t) { return t * STEP / 64 * kLineBytes + t * STEP % 64 * 2; }
};

__device__ __forceinline__ void tmem_st16(uint32_t taddr, const uint32_t (&v)[16]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], "
      "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16};" ::"r"(taddr),
      "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7]), "r"(v[8]), "r"(v[9]),
      "r"(v[10]), "r"(v[11]), "r"(v[12]), "r"(v[13]), "r"(v[14]), "r"(v[15])
      : "memory");
}
// 16 columns of this thread's lane, without waiting for them
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&v)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), "=r"(v[8]),
        "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
      : "r"(taddr)
      : "memory");
}

// D (+)= A B, bf16 terms: A in tensor memory (two k per 32-bit column), B MN-major in shared memory
__device__ __forceinline__ void umma_bf16_ta(uint32_t tmem_d, uint32_t tmem_a, uint64_t bdesc, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n"
      " .reg .pred p;\n"
      " setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n"
      "}\n" ::"r"(tmem_d),
      "r"(tmem_a), "l"(bdesc), "r"(idesc), "r"(acc)
      : "memory");
}

__device__ __forceinline__ void cp_async16(uint32_t dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void bulk_load(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(smem_u32(dst)),
               "l"(src), "r"(bytes), "r"(smem_u32(bar))
               : "memory");
}

// MN-major tile of 16-bit elements, 128-byte swizzle: 64 features of one column are 128 contiguous bytes, 8 columns a
// group of 1024 bytes, groups follow each other.  (A tile has one block of 64 features: no second offset.)
__device__ __forceinline__ uint64_t desc_mn_bf16(uint32_t smem_addr) {
  uint64_t d = 0;
  d |= (uint64_t)((smem_addr & 0x3FFFF) >> 4);
  d |= (uint64_t)(1024 >> 4) << 16;
  d |= (uint64_t)(1024 >> 4) << 32;
  d |= (uint64_t)1 << 46;
  d |= (uint64_t)2 << 61;  // SWIZZLE_128B
  return d;
}

struct Params {
  int nslab, n_tiles;
  const int32_t* prefix;     // [n_tiles + 1] chunks of the tiles before
  const int32_t* chunk_ptr;  // [n_tiles] where a tile's chunks start in tcol / bits
  const int32_t* tcol;       // [chunks x 64] source rows (a row of zeros where a slot is not used)
  const uint64_t* bits;      // [chunks x 256]
  const uint8_t* split;      // the three terms of X: row r at r * split_pitch bytes, nslab x lines x 128 bytes
  int64_t split_pitch;
  int per_cta, total;        // units
  float* pieces;             // [(tiles x nslab + CTAs)][256][N]
  int64_t rows, n_pieces;    // (checked by the GCNSA_DEBUG build)
  int* beyond;               // [0] set by split_rows: values the MMAs cannot take; moved to [1] for spmm_rest
};

// A CTA's run of units, tile by tile and slab by slab.
struct Item {
  int64_t chunk;  // where its first chunk is in tcol / bits
  int slab, len, piece;
};
struct Walk {
  int u, end, t, cnt, slab, k0;
  __device__ __forceinline__ void start(const Params& p) {
    u = blockIdx.x * p.per_cta;
    end = min(p.total, u + p.per_cta);
    t = cnt = slab = k0 = 0;
    if (u >= end) return;
    int lo = 0, hi = p.n_tiles - 1;  // the tile of unit u: the smallest t whose end lies behind u
    while (lo < hi) {
      const int mid = (lo + hi) >> 1;
      if ((int64_t)p.nslab * __ldg(p.prefix + mid + 1) > u) hi = mid;
      else lo = mid + 1;
    }
    t = lo;
    const int first = __ldg(p.prefix + t);
    cnt = __ldg(p.prefix + t + 1) - first;
    const int off = u - p.nslab * first;
    slab = off / cnt;
    k0 = off - slab * cnt;
  }
  __device__ __forceinline__ bool next(const Params& p, Item& it) {
    if (u >= end) return false;
    while (k0 >= cnt) {  // on to the next slab or the next tile that has chunks
      k0 = 0;
      if (++slab < p.nslab && cnt > 0) continue;
      slab = 0;
      ++t;
      cnt = __ldg(p.prefix + t + 1) - __ldg(p.prefix + t);
    }
    it.chunk = (int64_t)__ldg(p.chunk_ptr + t) + k0;
    it.slab = slab;
    it.len = min(cnt - k0, end - u);
    it.piece = t * p.nslab + slab + (int)blockIdx.x;
    u += it.len;
    k0 += it.len;
    return true;
  }
};

template <int N>
__global__ void __launch_bounds__(kThreads, 1) spmm_dense(const Params p) {
  using L = Lines<N>;
  constexpr int A_COL0 = 4 * N;     // tensor memory: two accumulators of 2 x N columns, then the A stages
  constexpr int ACC = 2 * N;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint64_t* full_a = reinterpret_cast<uint64_t*>(smem + L::BAR_OFF);  // A of the stage written (one arrival per expanding warp)
  uint64_t* full_b = full_a + kStagesA;                               // lines landed
  uint64_t* full_w = full_b + kStagesB;                               // bits landed (one arrival + bytes)
  // MMAs of a unit retired (one arrival per MMA warp): its A stage, its B stage and its accumulator change hands.  One
  // commit says it to all three (with one each the commits were what an MMA warp spent most of its time on).
  uint64_t* done = full_w + kStagesB;
  uint64_t* acc_empty = done + kStagesB;                                // accumulator read back (one per folding warp)
  uint64_t* drain = acc_empty + 2;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(drain + 2);
  int* abort_slot = reinterpret_cast<int*>(tmem_slot + 1);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

  if (threadIdx.x == 0) *abort_slot = tc_error_now();
  __syncthreads();
  if (*abort_slot != 0) {
    wait_for_predecessors();
    return;
  }
  if (threadIdx.x == 0) {
    for (int i = 0; i < kStagesA; ++i) mbar_init(&full_a[i], kRowWarps);
    for (int i = 0; i < kStagesB; ++i) {
      mbar_init(&full_b[i], 1);
      mbar_init(&full_w[i], 1);
      mbar_init(&done[i], 2);
    }
    for (int b = 0; b < 2; ++b) mbar_init(&acc_empty[b], kRowWarps);
    mbar_init(&drain[0], 1);
    mbar_init(&drain[1], 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32(tmem_slot)) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem_base = *tmem_slot;
  wait_for_predecessors();  // barriers and tensor memory are up; from here on global memory is read
  if (blockIdx.x == 0 && threadIdx.x == 0) {  // the word is 0 again before the next product's split_rows runs
    p.beyond[1] = p.beyond[0];
    p.beyond[0] = 0;
  }

  Walk walk;
  walk.start(p);
  Item it;

  const int n = max(0, min(p.total, (int)(blockIdx.x + 1) * p.per_cta) - (int)blockIdx.x * p.per_cta);

  if (warp < kExpandWarp0) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kRegsLoad));
    if (warp == 0 || warp == 7) {
      // ---------------- MMA issuers ----------------
      // The whole warp walks the units and one elected thread issues: loop counters, tensor-memory addresses and
      // descriptors are then known to be the same in all lanes and stay in uniform registers (with the walk inside the
      // elected branch every MMA moved its operands there first, 46 clocks each where the tensor pipe needs 32).
      // D fp32, A and B bf16, A K-major (tensor memory), B MN-major, 128 x N
      const int m = warp == 0 ? 0 : 1;
      const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | (1u << 16) | ((uint32_t)(N >> 3) << 17) | (8u << 24);
      const uint64_t b0 = desc_mn_bf16(smem_u32(smem));
      const uint32_t tm = __shfl_sync(0xffffffffu, tmem_base, 0);
      bool ok = true;
      int u = 0;
#pragma unroll 1
      for (; u < n; ++u) {
        const uint32_t sa = u % kStagesA, pa = (u / kStagesA) & 1, sb = u % kStagesB, pb = (u / kStagesB) & 1;
        const uint32_t b = u & 1, pe = ((u >> 1) & 1) ^ 1;
        // the three questions are asked at once (their answers take 30 clocks each); only a no leads to a wait
        const bool have_a = mbar_try_wait(&full_a[sa], pa), have_b = mbar_try_wait(&full_b[sb], pb),
                   have_acc = mbar_try_wait(&acc_empty[b], pe);
        if (!(have_a & have_b & have_acc))
          ok = mbar_wait(&acc_empty[b], pe, 24) && mbar_wait(&full_a[sa], pa, 25) && mbar_wait(&full_b[sb], pb, 26);
        if (!__all_sync(0xffffffffu, ok)) break;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const uint64_t bs = b0 + (uint64_t)((sb * L::STAGE) >> 4);
        const uint32_t a = tm + A_COL0 + sa * 64 + m * 32;
        const uint32_t d = tm + m * N + b * ACC;
        if (elect_one()) {
#pragma unroll
          for (int kk = 0; kk < 4; ++kk)
#pragma unroll
            for (int t = 2; t >= 0; --t)  // small terms first
              umma_bf16_ta(d, a + 8 * kk, bs + (uint64_t)((L::offset(t) + kk * 2048) >> 4), idesc, kk != 0 || t != 2);
          umma_commit(&done[sb]);
        }
        __syncwarp();
      }
      if (u < n && u > 0) {  // a wait ran out: the MMAs issued so far must have retired before tensor memory is given back
        if (elect_one()) umma_commit(&drain[m]);
        const long long t0 = clock64();
        while (!mbar_try_wait(&drain[m], 0) && clock64() - t0 < kSpinCycles) {
        }
      }
    } else {
      // ---------------- source rows: loading warp i takes units i, i + 6, ... ----------------
      // eight lanes take the 16-byte pieces of a line, the four groups of eight lanes 16 columns each
      const int q = lane >> 3, piece = lane & 7;
      int g = warp - kLoadWarp0, before = 0, at = 0;  // before: units before the item `it`
      bool have = walk.next(p, it), ok = true;
      auto seek = [&]() {  // the item of unit g
        while (have && g - before >= it.len) {
          before += it.len;
          have = walk.next(p, it);
        }
        at = g - before;
        return have;
      };
      int4 idx[4];
      auto indices = [&]() {
        const int4* src = reinterpret_cast<const int4*>(p.tcol + (it.chunk + at) * 64) + 4 * q;
#pragma unroll
        for (int i = 0; i < 4; ++i) idx[i] = __ldg(src + i);
      };
      if (seek()) indices();
      while (have) {
        const uint32_t s = g % kStagesB, ph = (g / kStagesB) & 1;
        ok = __all_sync(0xffffffffu, mbar_wait(&done[s], ph ^ 1, 22));
        if (!ok) break;
        uint8_t* stage = smem + s * L::STAGE;
        if (elect_one()) {
          mbar_expect_tx(&full_w[s], kBitBytes);
          bulk_load(stage + L::COUNT * kLineBytes, p.bits + (it.chunk + at) * 256, kBitBytes, &full_w[s]);
        }
        __syncwarp();
        const uint8_t* src = p.split + (int64_t)it.slab * L::COUNT * 128 + piece * 16;
        const uint32_t dst = smem_u32(stage + q * 2048);
#pragma unroll
        for (int i = 0; i < 16; ++i) {
          const int4& v = idx[i >> 2];
          int row = (i & 3) == 0 ? v.x : (i & 3) == 1 ? v.y : (i & 3) == 2 ? v.z : v.w;
#if GCNSA_DBG
          if (!dbg_in(&g_dbg_dense, row, 0, p.rows + 1, kDbgColumn)) row = (int)p.rows;  // the row of zeros
#endif
          const uint8_t* r = src + (int64_t)row * p.split_pitch;
#pragma unroll
          for (int line = 0; line < L::COUNT; ++line)
            cp_async16(dst + line * kLineBytes + (i >> 3) * 1024 + (i & 7) * 128 + ((piece ^ (i & 7)) << 4), r + line * 128);
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
        g += kLoadWarps;
        if (seek()) indices();  // on their way while the lines are
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // hand them to the tensor core
        __syncwarp();
        if (lane == 0) mbar_arrive(&full_b[s]);
      }
      if (!ok || tc_error_now() != 0) {  // the bit copies already issued land before the CTA exits
        const long long t0 = clock64();
        for (int gi = g - kLoadWarps; gi >= 0 && gi > g - 3 * kLoadWarps; gi -= kLoadWarps)
          while (!mbar_try_wait(&full_w[gi % kStagesB], (gi / kStagesB) & 1) && clock64() - t0 < kSpinCycles) {
          }
      }
    }
  } else if (warp < kFoldWarp0) {
    // ---------------- bits -> A ----------------
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kRegsExpand));
    const int mt = (warp - kExpandWarp0) >> 2, q = warp & 3, row = mt * 128 + q * 32 + lane;
    const uint32_t lanes = tmem_base + ((uint32_t)(32 * q) << 16) + A_COL0 + mt * 32;
    for (int g = 0; g < n; ++g) {
      // the stage of A is free when the MMAs of unit g - kStagesA have retired
      const uint32_t s = g % kStagesA, sb = g % kStagesB, pb = (g / kStagesB) & 1;
      const int e = g + kStagesB - kStagesA;
      uint64_t* freed = &done[e % kStagesB];
      const uint32_t pf = (e / kStagesB + 1) & 1;
      const bool have_w = mbar_try_wait(&full_w[sb], pb), have_a = mbar_try_wait(freed, pf);
      bool ok = have_w & have_a;
      if (!ok) ok = mbar_wait(&full_w[sb], pb, 27) && mbar_wait(freed, pf, 23);
      if (!__all_sync(0xffffffffu, ok)) break;
      const uint64_t w = *reinterpret_cast<const uint64_t*>(smem + sb * L::STAGE + L::COUNT * kLineBytes + row * 8);
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      // column j of A holds k = 2 j and 2 j + 1, bits j and j + 16 of a half of the word; a set bit lands on bit 14
      // of its bf16, which alone is the number 2 (the sums are halved on the way out: exact)
      uint32_t v[16];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const uint32_t half = (uint32_t)(w >> (32 * h));
#pragma unroll
        for (int j = 0; j < 16; ++j) v[j] = (j <= 14 ? half << (14 - j) : half >> 1) & 0x40004000u;
        tmem_st16(lanes + s * 64 + 16 * h, v);
      }
      asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      __syncwarp();
      if (lane == 0) mbar_arrive(&full_a[s]);
    }
  } else {
    // ---------------- accumulators -> running sums -> pieces ----------------
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kRegsFold));
    const int mt = (warp - kFoldWarp0) >> 2, q = warp & 3, row = mt * 128 + q * 32 + lane;
    const uint32_t lanes = tmem_base + ((uint32_t)(32 * q) << 16) + mt * N;
    float run[N];
    uint32_t g = 0;
    bool ok = true;
    while (ok && walk.next(p, it)) {
#pragma unroll
      for (int i = 0; i < N; ++i) run[i] = 0.f;
      for (int c = 0; c < it.len; ++c, ++g) {
        const uint32_t b = g & 1;
        ok = __all_sync(0xffffffffu, mbar_wait(&done[g % kStagesB], (g / kStagesB) & 1, 21));
        if (!ok) break;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
        for (int n0 = 0; n0 < N; n0 += 32) {  // two loads of 16 columns in flight
          uint32_t v[16], w[16];
          tmem_ld16(lanes + b * ACC + n0, v);
          if (n0 + 16 < N) tmem_ld16(lanes + b * ACC + n0 + 16, w);
          asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
          if (n0 + 32 >= N) {
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            __syncwarp();
            if (lane == 0) mbar_arrive(&acc_empty[b]);
          }
#pragma unroll
          for (int j = 0; j < 16; ++j) run[n0 + j] += __uint_as_float(v[j]);
          if (n0 + 16 < N) {
#pragma unroll
            for (int j = 0; j < 16; ++j) run[n0 + 16 + j] += __uint_as_float(w[j]);
          }
        }
      }
      if (!ok) break;
#if GCNSA_DBG
      if (!dbg_in(&g_dbg_dense, it.piece, 0, p.n_pieces, kDbgPartialSum)) continue;
#endif
      float4* dst = reinterpret_cast<float4*>(p.pieces + ((int64_t)it.piece * 256 + row) * N);
#pragma unroll
      for (int c = 0; c < N / 4; ++c)
        dst[c] = make_float4(0.5f * run[4 * c], 0.5f * run[4 * c + 1], 0.5f * run[4 * c + 2], 0.5f * run[4 * c + 3]);
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem_base) : "memory");
  }
}

// the upper halves of two words as a pair of bf16
__device__ __forceinline__ uint32_t upper_halves(float lo, float hi) {
  return __byte_perm(__float_as_uint(lo), __float_as_uint(hi), 0x7632);
}
// x minus its upper half: exact, and the result has at most 16 (then 8) significant bits
__device__ __forceinline__ uint32_t magnitude(const float4& v) {
  return max(max(__float_as_uint(v.x) & 0x7FFFFFFFu, __float_as_uint(v.y) & 0x7FFFFFFFu),
             max(__float_as_uint(v.z) & 0x7FFFFFFFu, __float_as_uint(v.w) & 0x7FFFFFFFu));
}
constexpr uint32_t kBeyond = (127u + 96u) << 23;  // the word of 2^96; Inf and NaN lie above
__device__ __forceinline__ float lower_part(float x) { return x - __uint_as_float(__float_as_uint(x) & 0xFFFF0000u); }

// The three bf16 terms of (xscale[i] times) every row, in the lines spmm_dense gathers; row n is zero (the row of slots
// that are not used).  A thread takes 8 features.
__global__ void __launch_bounds__(256)
split_rows(int64_t n, const float4* __restrict__ x, int64_t ldx4, int nvec, const float* __restrict__ xscale, int groups,
           int groups_per_slab, int step, int lines, uint4* __restrict__ out, int* __restrict__ beyond) {
  wait_for_predecessors();
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= (n + 1) * groups) return;
  const int64_t row = i / groups;
  const int gr = (int)(i - row * groups), slab = gr / groups_per_slab, in = gr - slab * groups_per_slab;
  float4 a = make_float4(0.f, 0.f, 0.f, 0.f), b = a;
  if (row < n) {
    const float4* src = x + row * ldx4;
    if (2 * gr < nvec) a = __ldg(src + 2 * gr);
    if (2 * gr + 1 < nvec) b = __ldg(src + 2 * gr + 1);
    if (xscale) {
      const float sc = __ldg(xscale + row);
      a.x *= sc; a.y *= sc; a.z *= sc; a.w *= sc;
      b.x *= sc; b.y *= sc; b.z *= sc; b.w *= sc;
    }
  }
  if (max(magnitude(a), magnitude(b)) >= kBeyond) *beyond = 1;
  const int slabs = groups / groups_per_slab;
  uint4* dst = out + (row * slabs + slab) * lines * 8 + in;
#pragma unroll
  for (int t = 0; t < 3; ++t) {
    dst[t * (step / 8)] = make_uint4(upper_halves(a.x, a.y), upper_halves(a.z, a.w), upper_halves(b.x, b.y), upper_halves(b.z, b.w));
    a = make_float4(lower_part(a.x), lower_part(a.y), lower_part(a.z), lower_part(a.w));
    b = make_float4(lower_part(b.x), lower_part(b.y), lower_part(b.z), lower_part(b.w));
  }
}

int sm_count() {
  static int n = 0;
  static std::once_flag once;
  std::call_once(once, [] {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n <= 0)
      n = 148;
  });
  return n;
}

// slabs of equal width, a multiple of 16 and at most 64 features
struct Slabs { int n, width, step, lines; };
Slabs slabs_of(int f) {
  Slabs s;
  s.n = (f + 63) / 64;
  s.width = ((f + s.n - 1) / s.n + 15) / 16 * 16;
  s.step = s.width <= 32 ? s.width : 64;
  s.lines = (3 * s.step + 63) / 64;
  return s;
}
struct Use { int tiles; int64_t chunks; const int32_t* prefix; };
Use use_of(const DensePlan& d, DenseUse use) {
  if (use == DenseUse::lossRows) return {d.loss_tiles, d.loss_tile_chunks, d.chunk_ptr};
  if (use == DenseUse::lossCols) return {d.n_tiles, d.n_loss_chunks, d.loss_ptr};
  return {d.n_tiles, d.n_chunks, d.chunk_ptr};
}
size_t pieces_bytes(const DensePlan& d, const Slabs& sl) {
  return ((size_t)d.n_tiles * sl.n + (size_t)sm_count()) * kDenseRows * sl.width * sizeof(float);
}

template <int N>
cudaError_t run(cudaStream_t s, int grid, const Params& p) {
  cudaError_t e = cudaFuncSetAttribute(spmm_dense<N>, cudaFuncAttributeMaxDynamicSharedMemorySize, Lines<N>::SMEM);
  if (e != cudaSuccess) return e;
  launch(spmm_dense<N>, grid, kThreads, Lines<N>::SMEM, s, p);
  note_launch();
  return cudaGetLastError();
}

}  // namespace

size_t spmm_planned_workspace(const DensePlan& d, int32_t f) {
  if (d.n_chunks == 0) return 0;
  const Slabs sl = slabs_of(f);
  return kPlannedHead + pieces_bytes(d, sl) + (size_t)(d.n_rows + 1) * sl.n * sl.lines * 128;
}

// What the three kernels of a product pull through the SMs: X once and its terms (split_rows), a unit's lines, slots and bits
// (spmm_dense), partial sums written and read, `rest_nnz` gathers, the result.
double spmm_planned_l1_bytes(const DensePlan& d, DenseUse use, int64_t n_rows, int64_t rest_nnz, int32_t f) {
  const Slabs sl = slabs_of(f);
  const Use us = use_of(d, use);
  const double units = (double)us.chunks * sl.n, line_bytes = (double)sl.lines * 128.0;
  const double pieces = ((double)us.tiles * sl.n + sm_count()) * kDenseRows * sl.width * 4.0;
  return (double)d.n_rows * (4.0 * f + sl.n * line_bytes) + units * (kDenseCols * (line_bytes + 4.0) + kBitBytes) + 2.0 * pieces +
         (double)rest_nnz * (4.0 * f + 4.0) + (double)n_rows * (4.0 * f + 16.0);
}

// -1: too many units to count in an int (the caller then gathers)
int launch_spmm_planned(void* stream, const DensePlan& d, DenseUse use, int64_t n_rows, const int32_t* rowptr,
                        const int32_t* col, const float* row_scale,
                        const float* src_scale, const float* x, int64_t ldx, int32_t f, int32_t epi, const float* aux,
                        int64_t ldaux, float* y, int64_t ldy, void* workspace, const SpmmBounds& bounds) {
  if (n_rows == 0 || f == 0) return 0;
  const Slabs sl = slabs_of(f);
  const Use us = use_of(d, use);
  const int64_t total = us.chunks * sl.n;
  if (total >= INT32_MAX / 2) return -1;
  SpmmBase base;
  int* beyond = (int*)workspace;
  float* pieces = (float*)((uint8_t*)workspace + kPlannedHead);
  base.pieces = pieces;
  base.pos = d.pos;
  base.prefix = us.prefix;
  base.nslab = sl.n;
  base.width = sl.width;
  base.per_cta = 1;
  if (total > 0) {
    cudaStream_t s = (cudaStream_t)stream;
    const int sms = sm_count();
    uint8_t* split = (uint8_t*)pieces + pieces_bytes(d, sl);
    const int gps = sl.width / 8, groups = gps * sl.n;
    const int64_t threads = (d.n_rows + 1) * groups;
    launch(split_rows, (unsigned)((threads + 255) / 256), 256, 0, s, d.n_rows, reinterpret_cast<const float4*>(x), ldx / 4,
                                                                 (f + 3) / 4, src_scale, groups, gps, sl.step, sl.lines,
                                                                 reinterpret_cast<uint4*>(split), beyond);
    note_launch();
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return (int)e;
    Params p;
    p.nslab = sl.n; p.n_tiles = us.tiles;
    p.prefix = us.prefix; p.chunk_ptr = d.chunk_ptr; p.tcol = d.tcol; p.bits = d.bits;
    p.total = (int)total;
    p.per_cta = (int)((total + sms - 1) / sms);
    p.pieces = pieces;
    p.rows = d.n_rows;
    p.n_pieces = base.n_pieces = (int64_t)d.n_tiles * sl.n + sms;
    p.beyond = beyond;
    base.beyond = beyond + 1;
    base.all_rowptr = rowptr;
    base.all_col = col;
    base.all_nnz = bounds.nnz;
    p.split = split;
    p.split_pitch = (int64_t)sl.n * sl.lines * 128;
    base.per_cta = p.per_cta;
    if (p.per_cta > 1 && total * p.per_cta < (1LL << 32)) base.magic = (unsigned)(((1ULL << 32) + p.per_cta - 1) / p.per_cta);
    const int grid = (int)((total + p.per_cta - 1) / p.per_cta);
    if (sl.width == 16) e = run<16>(s, grid, p);
    else if (sl.width == 32) e = run<32>(s, grid, p);
    else if (sl.width == 48) e = run<48>(s, grid, p);
    else e = run<64>(s, grid, p);
    if (e != cudaSuccess) return (int)e;
  }
  return launch_spmm_rest(stream, n_rows, d.r_rowptr, use == DenseUse::lossCols ? d.r_mid : d.r_rowptr + 1, d.r_col,
                          row_scale, src_scale, use == DenseUse::lossRows ? d.rm_order : d.r_order,
                          use == DenseUse::lossRows ? d.rm_n_long : d.r_n_long, x, ldx, f, epi, aux, ldaux, y, ldy, base,
                          SpmmBounds{bounds.mat_rows, bounds.src_rows, d.r_nnz});
}

int debug_word_dense(unsigned long long* out, bool clear) {
  *out = 0ull;
#if GCNSA_DBG
  cudaError_t e = cudaMemcpyFromSymbol(out, g_dbg_dense, sizeof(*out));
  if (e == cudaSuccess && clear) {
    const unsigned long long zero = 0ull;
    e = cudaMemcpyToSymbol(g_dbg_dense, &zero, sizeof(zero));
  }
  return (int)e;
#else
  (void)clear;
  return 0;
#endif
}

int tc_status(int* out) {
  int v = 0, w = 0;
  cudaError_t e = cudaMemcpyFromSymbol(&v, g_tc_error, sizeof(int));
  if (e != cudaSuccess) return (int)e;
  const int r = tc_status_gemm(&w);
  *out = w ? w : v;
  return r;
}
int tc_clear() {
  const int zero = 0;
  cudaError_t e = cudaMemcpyToSymbol(g_tc_error, &zero, sizeof(int));
  return e != cudaSuccess ? (int)e : tc_clear_gemm();
}

}  // namespace gcnsa
