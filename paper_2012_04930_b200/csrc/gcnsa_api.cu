// C-ABI of libgcnsa: handles, device memory, and the order in which the kernels
// of one forward / backward / step are enqueued.
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <cstring>
#include <mutex>
#include <new>
#include <string>
#include <thread>
#include <vector>

#include "internal.h"
#include "parts.h"

namespace gcnsa {

static thread_local std::string g_err;
static std::atomic<int64_t> g_launches{0};

int fail(int code, const std::string& detail) {
  g_err = detail;
  return code;
}
void note_launch(int n) { g_launches.fetch_add(n, std::memory_order_relaxed); }
static std::atomic<int64_t> g_gemm_tc{0}, g_gemm_fallback{0};
void note_gemm_path(bool tensor_core) { (tensor_core ? g_gemm_tc : g_gemm_fallback).fetch_add(1, std::memory_order_relaxed); }

static int cuda_fail(cudaError_t e, const char* what) {
  return fail(GCNSA_ERR_CUDA, std::string(what) + ": " + cudaGetErrorString(e));
}
#define CK(call)                                          \
  do {                                                    \
    cudaError_t e_ = (call);                              \
    if (e_ != cudaSuccess) return cuda_fail(e_, #call);   \
  } while (0)
#define CKL(call)                                                       \
  do {                                                                  \
    int e_ = (call);                                                    \
    if (e_ != 0) return cuda_fail((cudaError_t)e_, #call);              \
  } while (0)

static int check_device(const gcnsa_env* env) {
  if (!env) return fail(GCNSA_ERR_ARG, "env is NULL");
  if ((env->alloc == nullptr) != (env->free == nullptr)) return fail(GCNSA_ERR_ARG, "alloc and free must come together");
  int count = 0;
  cudaError_t e = cudaGetDeviceCount(&count);
  if (e != cudaSuccess || count == 0) {
    cudaGetLastError();
    return fail(GCNSA_ERR_CUDA, "no CUDA device: this library has no CPU fallback");
  }
  if (env->device < 0 || env->device >= count) return fail(GCNSA_ERR_ARG, "device index out of range");
  CK(cudaSetDevice(env->device));
  int major = 0;  // (one attribute: all properties of a device take 2.8 ms to ask for)
  CK(cudaDeviceGetAttribute(&major, cudaDevAttrComputeCapabilityMajor, env->device));
  if (major != 10) return fail(GCNSA_ERR_UNSUPPORTED_ARCH, "kernels are built for sm_100a only");
  return GCNSA_OK;
}

}  // namespace gcnsa

using namespace gcnsa;

extern "C" int64_t gcnsa_launch_count(void);

// Activations, work buffers and reduction scratch of one pass over a partition.  Lane 0 serves the calls that go
// partition by partition; a recorded epoch runs several partitions at once, one per lane (epoch_lanes).
struct Lane {
  float* H[GCNSA_MAX_LAYERS + 1] = {nullptr};  // H[l], l >= 1
  float* S[GCNSA_MAX_LAYERS] = {nullptr};      // A_hat H^{l-1} of layers that aggregate first
  float *tmp_a = nullptr, *tmp_b = nullptr, *dlogits = nullptr;
  float* ce_sums = nullptr;        // partial column sums of dlogits (the last layer's bias gradient), where the softmax makes them
  void *ws = nullptr, *sc = nullptr;
  float* ce_part = nullptr;        // the softmax kernel's partial sums of the loss
  void* dw = nullptr;              // workspace of the planned sparse products
  const float* s0_used = nullptr;  // A_hat H^0 the latest forward used (the cached one or S[0])
};

struct gcnsa_model {
  Env env;
  gcnsa_model_opts o{};
  int32_t L = 0, m = 0;
  int64_t n_max = 0, count = 0;  // count = floats in the flat parameter buffer
  int64_t w_off[GCNSA_MAX_LAYERS], b_off[GCNSA_MAX_LAYERS], w_ld[GCNSA_MAX_LAYERS];
  bool transform_first[GCNSA_MAX_LAYERS];
  float *theta = nullptr, *gsum = nullptr, *am = nullptr, *av = nullptr;
  // parameter-averaging mode: Adam moments per partition ([m x count]) and the running mean of the partitions' parameters
  float *am_parts = nullptr, *av_parts = nullptr, *theta_acc = nullptr;
  int32_t state_p = 0;
  bool all_rows_once = false;  // set by gcnsa_evaluate: the next forward computes every logit row
  double* adam_state = nullptr;  // device: step count t and the two bias corrections of Adam
  // recorded epoch (epoch_graph): valid for one partitions object and one loss pointer
  cudaGraphExec_t graph_exec = nullptr;
  uint64_t graph_parts_uid = 0;
  const void* graph_loss = nullptr;
  int graph_kernels = 0;  // kernel launches one replay stands for
  bool graph_off = false;
  // cache_ax: A_hat X of every partition of one partitions object, kept while the feature rows stay the same
  std::vector<float*> ax;
  std::vector<int64_t> ax_version;  // x_version of the partition the product was computed from (0 = none yet)
  uint64_t ax_uid = 0;
  std::vector<Lane> lanes;        // at least one
  mutable std::mutex pack;        // gcnsa_model_get packs rows in the work buffer of lane 0: one caller at a time
  float* gparts = nullptr;        // [m x count]: the gradient of every partition of an epoch; NULL: they go into gsum
  float* loss_parts = nullptr;
  // evaluation buffers (allocated on first gcnsa_evaluate)
  int32_t *ev_pred = nullptr, *ev_hits = nullptr;
  uint8_t* ev_mask = nullptr;
  size_t ws_bytes = 0, sc_bytes = 0, dw_bytes = 0;
  int beside = 1;  // partitions a recorded epoch may work on at once (whether it does or not: results do not depend on it)
  int64_t ld_max = 0;
  int32_t last_forward = -1, accumulated = 0;
  int64_t last_n = 0;
  int64_t t = 0;
  std::vector<void*> owned;
  void* dalloc(size_t bytes) {
    void* p = env.alloc(bytes);
    if (p) owned.push_back(p);
    return p;
  }
  // optional per-kernel timing
  struct Rec { int cat; double bytes, flops, l1, bytes_val; int64_t launches; };
  bool prof_on = false;
  std::vector<cudaEvent_t> ev;  // pairs, reused
  std::vector<Rec> recs;
  int64_t launches_mark = 0;
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
  void prof_end(int cat, double bytes, double flops, double l1 = -1.0, double bytes_val = -1.0) {
    if (!prof_on) return;
    cudaEventRecord(ev[recs.size() * 2 + 1], env.stream());
    recs.push_back({cat, bytes, flops, l1 < 0.0 ? bytes : l1, bytes_val < 0.0 ? bytes : bytes_val,
                    gcnsa_launch_count() - launches_mark});
  }
};

// Memory accounting of one sparse product over `rows` result rows, `nnz` stored entries and `n_src` source rows
// that are referenced, at width f.  bytes: what must cross HBM once (row pointers, column indices, values - none
// when the normalization is factored out: then one scale per row -, one read of the source rows, one write of the
// result, one read of a ReLU mask).  l1: what the SMs pull through the L1 data path: the same, except that every
// stored entry gathers its own source row (4 f nnz instead of 4 f n_src).
// bytes_val: `bytes` with 8 bytes per stored entry (index + value) whether or not the kernel reads values.
struct SpmmCost { double bytes, l1, flops, bytes_val; };
static SpmmCost spmm_cost(int64_t rows, int64_t n_src, int64_t nnz, int64_t f, bool values, bool mask = false) {
  const double idx = 4.0 * (double)(rows + 1) + (values ? 8.0 * (double)nnz : 4.0 * (double)nnz + 4.0 * (double)rows);
  const double out = 4.0 * (double)f * (double)rows * (mask ? 2.0 : 1.0);
  SpmmCost c;
  c.bytes = idx + 4.0 * (double)f * (double)n_src + out;
  c.l1 = idx + 4.0 * (double)f * (double)nnz + out;
  c.flops = 2.0 * (double)nnz * (double)f;
  c.bytes_val = 4.0 * (double)(rows + 1) + 8.0 * (double)nnz + 4.0 * (double)f * (double)n_src + out;
  return c;
}
static double gemm_bytes(int64_t m, int64_t n, int64_t k) { return 4.0 * ((double)m * k + (double)k * n + (double)m * n); }
#define PROF(M, cat, bytes, flops, call) \
  do {                                   \
    (M)->prof_begin();                   \
    CKL(call);                           \
    (M)->prof_end(cat, bytes, flops);    \
  } while (0)
#define PROF_SPMM(M, cost, call)                             \
  do {                                                       \
    const SpmmCost c_ = (cost);                              \
    (M)->prof_begin();                                       \
    CKL(call);                                               \
    (M)->prof_end(0, c_.bytes, c_.flops, c_.l1, c_.bytes_val); \
  } while (0)

extern "C" {

const char* gcnsa_strerror(int code) {
  switch (code) {
    case GCNSA_OK: return "ok";
    case GCNSA_ERR_ARG: return "invalid argument";
    case GCNSA_ERR_NOT_SYMMETRIC: return "graph is not symmetric";
    case GCNSA_ERR_SELF_LOOP_OR_DUP: return "graph has a self-loop or a repeated edge";
    case GCNSA_ERR_LABEL_RANGE: return "label or partition id out of range";
    case GCNSA_ERR_OOM: return "out of memory";
    case GCNSA_ERR_ORDER: return "calls in the wrong order";
    case GCNSA_ERR_CUDA: return "CUDA error";
    case GCNSA_ERR_UNSUPPORTED_ARCH: return "device is not sm_100";
    case GCNSA_ERR_TOO_LARGE: return "partition exceeds int32 indexing";
    default: return "unknown error";
  }
}
const char* gcnsa_last_error(void) { return g_err.c_str(); }
int64_t gcnsa_launch_count(void) { return g_launches.load(); }
int gcnsa_gemm_path_counts(int64_t* tensor_core, int64_t* fp32_fallback) {
  if (!tensor_core || !fp32_fallback) return fail(GCNSA_ERR_ARG, "NULL argument");
  *tensor_core = g_gemm_tc.load();
  *fp32_fallback = g_gemm_fallback.load();
  return GCNSA_OK;
}
void gcnsa_model_opts_default(gcnsa_model_opts* o) {
  if (!o) return;
  std::memset(o, 0, sizeof(*o));
  o->n_layers = 2;
  o->use_bias = 1;
  o->lr = 0.02f; o->beta1 = 0.9f; o->beta2 = 0.999f; o->eps = 1e-8f;
  o->gemm_mode = GCNSA_GEMM_TF32X3;
  o->agg_mode = GCNSA_AGG_GRAD_AVG;
  o->loss_rows_only = 1;
  o->epoch_graph = 1;
  o->factored_norm = 1;
  o->cache_ax = 0;
}

// ------------------------------------------------------------------ parts ---
int gcnsa_parts_destroy(gcnsa_parts* parts) {
  if (!parts) return GCNSA_OK;
  cudaStreamSynchronize(parts->env.stream());
  if (parts->copy_stream) {
    cudaStreamSynchronize(parts->copy_stream);
    cudaStreamDestroy(parts->copy_stream);
  }
  for (cudaEvent_t e : parts->ready) cudaEventDestroy(e);
  for (cudaEvent_t e : parts->consumed) cudaEventDestroy(e);
  for (void* p : parts->owned) parts->env.release(p);
  delete parts;
  return GCNSA_OK;
}

static int upload(gcnsa_parts* P, void** dst, const void* src, size_t bytes) {
  *dst = P->dalloc(bytes);
  if (!*dst) return fail(GCNSA_ERR_OOM, "device allocation failed");
  if (bytes) CK(cudaMemcpyAsync(*dst, src, bytes, cudaMemcpyHostToDevice, P->env.stream()));
  return GCNSA_OK;
}

static int build_failed(gcnsa_parts* P, int rc) {
  std::string keep = g_err;
  gcnsa_parts_destroy(P);
  g_err = keep;
  return rc;
}

int gcnsa_build_partitions(const gcnsa_env* env, const gcnsa_graph* g, const gcnsa_part_opts* opts, gcnsa_parts** out) {
  if (!out) return fail(GCNSA_ERR_ARG, "out is NULL");
  *out = nullptr;
  int rc = check_build_args(g, opts);
  if (rc) return rc;
  HostBuild hb;
  const bool on_host = opts->builder == GCNSA_BUILD_HOST;
  if (on_host) {
    rc = build_host(g, opts, &hb);
    if (rc) return rc;
  }
  rc = check_device(env);
  if (rc) {
    // without a usable device an invalid graph is still reported as such (checked on the host cores)
    if (!on_host) {
      const std::string keep = g_err;
      const int v = validate_graph_host(g);
      if (v) return v;
      g_err = keep;
    }
    return rc;
  }
  gcnsa_parts* P = new (std::nothrow) gcnsa_parts();
  if (!P) return fail(GCNSA_ERR_OOM, "host allocation failed");
  P->env.e = *env;
  P->m = opts->m; P->f = g->f; P->c = g->c; P->n = g->n; P->ldx = GCNSA_LD(g->f);
  P->builder = opts->builder;
  static std::atomic<uint64_t> next_uid{1};
  P->uid = next_uid.fetch_add(1);
  if (!on_host) {
    try {
      P->x_version.assign((size_t)opts->m, 1);
      rc = build_device(P, g, opts);
    } catch (const std::bad_alloc&) {  // (the builder has joined its threads and handed its scratch back)
      rc = fail(GCNSA_ERR_OOM, "host allocation failed");
    }
    if (rc) return build_failed(P, rc);
    *out = P;
    return GCNSA_OK;
  }
  P->x_version.assign((size_t)opts->m, 1);
  P->part.swap(hb.part);
  P->parts.resize((size_t)opts->m);
  cudaStream_t s = P->env.stream();
  std::vector<float> xs;
  std::vector<int32_t> ys, deg;
  std::vector<uint8_t> ms;
  for (int32_t p = 0; p < opts->m && rc == GCNSA_OK; ++p) {
    HostPart& hp = hb.parts[p];
    DevPart& d = P->parts[p];
    d.info.n_owned = hp.n_owned; d.info.n_halo = hp.n_halo; d.info.n = hp.n; d.info.nnz = hp.nnz;
    d.info.nts = hp.nts; d.info.n_train = hp.n_train; d.info.max_depth = hp.max_depth;
    d.n_long = hp.n_long; d.t_n_long = hp.t_n_long;
    d.tm_n_long = hp.tm_n_long; d.tm_nnz = (int64_t)hp.tm_col.size();
    d.m_n_long = hp.m_n_long; d.m_nnz = hp.m_nnz;
    d.members.swap(hp.members);
    d.depth.swap(hp.depth);
    P->n_max = std::max(P->n_max, hp.n);
    const size_t n = (size_t)hp.n, nnz = (size_t)hp.nnz;
    // features, labels and mask in partition order (pad columns zero)
    xs.assign(n * (size_t)P->ldx, 0.f);
    ys.resize(n); ms.resize(n); deg.resize(n);
    {
      const int64_t chunk = 2048, n_chunks = ((int64_t)n + chunk - 1) / chunk;
      std::atomic<int64_t> next{0};
      auto work = [&] {
        for (;;) {
          const int64_t ci = next.fetch_add(1);
          if (ci >= n_chunks) break;
          for (int64_t i = ci * chunk; i < std::min<int64_t>((int64_t)n, (ci + 1) * chunk); ++i)
            std::memcpy(&xs[(size_t)i * P->ldx], g->x + d.members[i] * g->ldx, sizeof(float) * (size_t)g->f);
        }
      };
      int nt = (int)std::min<int64_t>(std::max(1u, std::thread::hardware_concurrency()), 16);
      std::vector<std::thread> th;
      for (int t = 1; t < nt; ++t) th.emplace_back(work);
      work();
      for (auto& t : th) t.join();
    }
    for (size_t i = 0; i < n; ++i) {
      ys[i] = g->y[d.members[i]];
      const bool carries = opts->loss_on_halo || (int64_t)i < hp.n_owned;
      ms[i] = (carries && g->train_mask[d.members[i]]) ? 1 : 0;
      deg[i] = hp.rowptr[i + 1] - hp.rowptr[i];
    }
    void* ddeg = nullptr;
#define UP(field, vec, type) if (rc == GCNSA_OK) rc = upload(P, (void**)&d.field, vec.data(), vec.size() * sizeof(type))
    UP(rowptr, hp.rowptr, int32_t); UP(col, hp.col, int32_t); UP(t_rowptr, hp.t_rowptr, int32_t);
    UP(t_col, hp.t_col, int32_t); UP(order, hp.order, int32_t); UP(t_order, hp.t_order, int32_t);
    UP(x, xs, float); UP(y, ys, int32_t); UP(mask, ms, uint8_t);
    UP(m_order, hp.m_order, int32_t);
    UP(tm_rowptr, hp.tm_rowptr, int32_t); UP(tm_col, hp.tm_col, int32_t); UP(tm_order, hp.tm_order, int32_t);
#undef UP
    if (rc == GCNSA_OK) rc = upload(P, &ddeg, deg.data(), n * sizeof(int32_t));
    if (rc == GCNSA_OK) {
      d.val = (float*)P->dalloc(std::max<size_t>(nnz, 1) * sizeof(float));
      d.t_val = (float*)P->dalloc(std::max<size_t>(nnz, 1) * sizeof(float));
      d.tm_val = (float*)P->dalloc(std::max<size_t>((size_t)d.tm_nnz, 1) * sizeof(float));
      d.dinv = (float*)P->dalloc(std::max<size_t>(n, 1) * sizeof(float));
      if (!d.val || !d.t_val || !d.tm_val || !d.dinv) rc = fail(GCNSA_ERR_OOM, "device allocation failed");
    }
    if (rc == GCNSA_OK) {
      // entry (i, j) of A_hat and entry (j, i) of its transpose are both
      // 1 / sqrt(d_i d_j) with d the row lengths of A + I: one degree array serves both
      int e1 = launch_normalize(s, hp.n, d.rowptr, d.col, (const int32_t*)ddeg, d.val);
      int e2 = launch_normalize(s, hp.n, d.t_rowptr, d.t_col, (const int32_t*)ddeg, d.t_val);
      if (!e2) e2 = launch_normalize(s, hp.n, d.tm_rowptr, d.tm_col, (const int32_t*)ddeg, d.tm_val);
      if (!e2) e2 = launch_inv_sqrt_degree(s, hp.n, (const int32_t*)ddeg, d.dinv);
      if (e1 || e2) rc = cuda_fail((cudaError_t)(e1 ? e1 : e2), "normalize");
    }
    if (rc == GCNSA_OK) rc = build_dense_plan(P, d, order_window_rows(opts->order_window, hp.n));
    // host staging vectors are reused: wait for the copies of this partition
    if (rc == GCNSA_OK) {
      cudaError_t e = cudaStreamSynchronize(s);
      if (e != cudaSuccess) rc = cuda_fail(e, "cudaStreamSynchronize");
    }
  }
  if (rc != GCNSA_OK) return build_failed(P, rc);
  *out = P;
  return GCNSA_OK;
}

int gcnsa_parts_count(const gcnsa_parts* parts) { return parts ? parts->m : GCNSA_ERR_ARG; }

int gcnsa_parts_info(const gcnsa_parts* parts, int32_t p, gcnsa_part_info* out) {
  if (!parts || !out || p < 0 || p >= parts->m) return fail(GCNSA_ERR_ARG, "bad partition index or NULL");
  *out = parts->parts[p].info;
  return GCNSA_OK;
}

int gcnsa_parts_assignment(const gcnsa_parts* parts, int32_t* part_host) {
  if (!parts || !part_host) return fail(GCNSA_ERR_ARG, "NULL argument");
  std::memcpy(part_host, parts->part.data(), parts->part.size() * sizeof(int32_t));
  return GCNSA_OK;
}

int gcnsa_parts_export(const gcnsa_parts* parts, int32_t p, const gcnsa_part_host* dst) {
  if (!parts || !dst || p < 0 || p >= parts->m) return fail(GCNSA_ERR_ARG, "bad partition index or NULL");
  const DevPart& d = parts->parts[p];
  cudaStream_t s = parts->env.stream();
  const size_t n = (size_t)d.info.n, nnz = (size_t)d.info.nnz;
#define DOWN(field, count, type) \
  if (dst->field) CK(cudaMemcpyAsync(dst->field, d.field, (count) * sizeof(type), cudaMemcpyDeviceToHost, s))
  DOWN(rowptr, n + 1, int32_t); DOWN(col, nnz, int32_t); DOWN(val, nnz, float);
  DOWN(t_rowptr, n + 1, int32_t); DOWN(t_col, nnz, int32_t); DOWN(t_val, nnz, float);
#undef DOWN
  if (dst->members) std::memcpy(dst->members, d.members.data(), n * sizeof(int64_t));
  if (dst->depth) std::memcpy(dst->depth, d.depth.data(), d.depth.size() * sizeof(int32_t));
  CK(cudaStreamSynchronize(s));
  return GCNSA_OK;
}

int gcnsa_parts_export_schedule(const gcnsa_parts* parts, int32_t p, gcnsa_part_schedule_info* info,
                                const gcnsa_part_schedule_host* dst) {
  if (!parts || p < 0 || p >= parts->m) return fail(GCNSA_ERR_ARG, "bad partition index or NULL");
  const DevPart& d = parts->parts[p];
  if (info) {
    info->n_long = d.n_long; info->t_n_long = d.t_n_long; info->m_n_long = d.m_n_long; info->tm_n_long = d.tm_n_long;
    info->m_nnz = d.m_nnz; info->tm_nnz = d.tm_nnz;
  }
  if (!dst) return GCNSA_OK;
  cudaStream_t s = parts->env.stream();
  const size_t n = (size_t)d.info.n;
#define DOWN(field, count, type) \
  if (dst->field && (count)) CK(cudaMemcpyAsync(dst->field, d.field, (count) * sizeof(type), cudaMemcpyDeviceToHost, s))
  DOWN(order, n, int32_t); DOWN(t_order, n, int32_t); DOWN(m_order, (size_t)d.info.n_train, int32_t);
  DOWN(tm_rowptr, n + 1, int32_t); DOWN(tm_col, (size_t)d.tm_nnz, int32_t); DOWN(tm_order, n, int32_t);
  DOWN(mask, n, uint8_t); DOWN(y, n, int32_t);
#undef DOWN
  CK(cudaStreamSynchronize(s));
  return GCNSA_OK;
}

int gcnsa_parts_get_features(const gcnsa_parts* parts, int32_t p, float* x_host) {
  if (!parts || !x_host || p < 0 || p >= parts->m) return fail(GCNSA_ERR_ARG, "bad partition index or NULL");
  const DevPart& d = parts->parts[p];
  if (d.info.n == 0) return GCNSA_OK;
  CK(cudaMemcpy2DAsync(x_host, (size_t)parts->f * sizeof(float), d.x, (size_t)parts->ldx * sizeof(float),
                       (size_t)parts->f * sizeof(float), (size_t)d.info.n, cudaMemcpyDeviceToHost, parts->env.stream()));
  CK(cudaStreamSynchronize(parts->env.stream()));
  return GCNSA_OK;
}

int gcnsa_parts_set_features(gcnsa_parts* parts, int32_t p, const float* x_host) {
  if (!parts || !x_host || p < 0 || p >= parts->m) return fail(GCNSA_ERR_ARG, "bad partition index or NULL");
  DevPart& d = parts->parts[p];
  CK(cudaMemcpy2DAsync(d.x, (size_t)parts->ldx * sizeof(float), x_host, (size_t)parts->f * sizeof(float),
                       (size_t)parts->f * sizeof(float), (size_t)d.info.n, cudaMemcpyHostToDevice, parts->env.stream()));
  parts->x_version[p] += 1;
  return GCNSA_OK;
}

}  // extern "C"

// ------------------------------------------------------------------ model ---
extern "C" {

int gcnsa_model_destroy(gcnsa_model* model) {
  if (!model) return GCNSA_OK;
  cudaStreamSynchronize(model->env.stream());
  for (void* p : model->owned) model->env.release(p);
  for (cudaEvent_t e : model->ev) cudaEventDestroy(e);
  if (model->graph_exec) cudaGraphExecDestroy(model->graph_exec);
  delete model;
  return GCNSA_OK;
}

static int copy_param(const gcnsa_model* M, float* base, int32_t layer, bool is_w, void* host, size_t bytes, bool to_host) {
  const int64_t rows = is_w ? M->o.dims[layer] : 1, cols = M->o.dims[layer + 1];
  if (bytes != (size_t)(rows * cols) * sizeof(float)) return fail(GCNSA_ERR_ARG, "byte count does not match the tensor");
  float* d = base + (is_w ? M->w_off[layer] : M->b_off[layer]);
  const size_t dpitch = (size_t)(is_w ? M->w_ld[layer] : cols) * sizeof(float), hpitch = (size_t)cols * sizeof(float);
  if (to_host) CK(cudaMemcpy2DAsync(host, hpitch, d, dpitch, hpitch, (size_t)rows, cudaMemcpyDeviceToHost, M->env.stream()));
  else CK(cudaMemcpy2DAsync(d, dpitch, host, hpitch, hpitch, (size_t)rows, cudaMemcpyHostToDevice, M->env.stream()));
  CK(cudaStreamSynchronize(M->env.stream()));
  return GCNSA_OK;
}

// How many partitions a recorded epoch works on at once: up to kMaxLanes while a partition has at most kLaneNnz stored
// entries.  The kernels of such a partition are microseconds long and leave most of the chip idle, so the epoch is a
// chain of launch latencies that the branches overlap (2 000 vertices, 2 partitions: 145 -> 83 us per epoch; 20 000
// vertices, 4 partitions: 403 -> 224 us; 58 241 vertices, 1.9 M entries in each of 3 partitions: 835 -> 684 us).  At
// 20.8 M entries per partition every sparse product fills the chip by itself and two of them at once evict each
// other's source rows from L1 and L2 (233 K vertices, 5 partitions: 7.1 ms with one lane, 8.1 with two, 9.0 with
// five); at 10 M entries two lanes gain 1 % and four lose 3 % (2.45 M vertices), which does not pay for the memory.
// What counts beside the entries is the rows: a lane is activations and work buffers for all of them.  Eight partitions
// without locality, one lane against eight: 8 000 rows of 8 entries, 64 wide (7 MB a lane) 587 -> 251 us per epoch, 64 000
// rows (58 MB) 1 161 -> 954; three layers of 256, 32 000 rows (156 MB) 2 727 -> 2 508, 64 000 rows (294 MB) 4 871 -> 4 800,
// 125 000 rows of 4 entries (556 MB) 9 101 -> 9 407, 250 000 rows (1.1 GB) 18 010 -> 18 240.  So the lanes after the first
// together take at most 1 GB: seven of 146 MB, three of 294 MB, none of more than 1 GB.  Lanes need a gradient buffer per
// partition; models with as many partitions and parameters that these would pass kGradBytes add into one sum instead, one
// partition after the other.
constexpr int64_t kMaxLanes = 8, kLaneNnz = 4 << 20;
constexpr size_t kLaneBytes = (size_t)1 << 30, kGradBytes = (size_t)64 << 20;
static int epoch_lanes(const gcnsa_model* M, const gcnsa_parts* parts, size_t lane_bytes) {
  int64_t nnz_max = 0;
  for (const DevPart& d : parts->parts) nnz_max = std::max<int64_t>(nnz_max, d.info.nnz);
  if (!M->o.epoch_graph || M->env.stream() == nullptr || nnz_max > kLaneNnz || !M->gparts) return 1;  // (the default stream records nothing)
  return (int)std::min<int64_t>(std::min<int64_t>(parts->m, kMaxLanes), 1 + (int64_t)(kLaneBytes / lane_bytes));
}

// Whether partitions are small enough that several are worked on at once (epoch_lanes: where kernels leave room beside them).
static bool beside(const gcnsa_parts* P) {
  int64_t nnz_max = 0;
  for (const DevPart& d : P->parts) nnz_max = std::max<int64_t>(nnz_max, d.info.nnz);
  return nnz_max <= kLaneNnz;
}
// Whether the passes of a recorded epoch have branches: while the chain of launches is the time.  A pass of two layers goes from
// 16 launches in a row to 11: ten epochs on 2 000 vertices 702 -> 640 us, on 20 000 vertices (partitions of 5 500 rows) 1 548 ->
// 1 486 us, partitions of 21 400 rows alike (3 085 -> 3 069 us), 51 400 rows (a hidden layer of 222) 1 000 -> 1 013.
constexpr int64_t kBranchRows = 16384;
static bool branches(const gcnsa_parts* P) { return beside(P) && P->n_max <= kBranchRows && ce_by_groups(P->c); }

// one lane's buffers; *bytes (nullable) grows by what was asked for
static bool alloc_lane(gcnsa_model* M, Lane& W, size_t act, size_t* bytes_out = nullptr) {
  auto get = [&](size_t bytes) {
    if (bytes_out) *bytes_out += bytes;
    return (float*)M->dalloc(bytes);
  };
  W.tmp_a = get(act);
  W.tmp_b = get(act);
  W.dlogits = get((size_t)M->n_max * GCNSA_LD(M->o.dims[M->L]) * sizeof(float));
  W.ce_sums = get(std::max<size_t>(ce_sums_scratch(M->o.dims[M->L]), 256));
  W.ws = get(std::max<size_t>(M->ws_bytes, 256));
  W.sc = get(std::max<size_t>(M->sc_bytes, 256));
  W.ce_part = get(std::max<size_t>(softmax_ce_scratch(M->n_max), 256));
  bool ok = W.tmp_a && W.tmp_b && W.dlogits && W.ce_sums && W.ws && W.sc && W.ce_part;
  for (int l = 0; l < M->L && ok; ++l) {
    W.H[l + 1] = get((size_t)M->n_max * GCNSA_LD(M->o.dims[l + 1]) * sizeof(float));
    ok = W.H[l + 1] != nullptr;
    if (ok && !M->transform_first[l]) {
      W.S[l] = get((size_t)M->n_max * GCNSA_LD(M->o.dims[l]) * sizeof(float));
      ok = W.S[l] != nullptr;
    }
  }
  return ok;
}

int gcnsa_model_create(const gcnsa_env* env, const gcnsa_parts* parts, const gcnsa_model_opts* opts,
                       const float* const* w0, const float* const* b0, gcnsa_model** out) {
  if (!out) return fail(GCNSA_ERR_ARG, "out is NULL");
  *out = nullptr;
  if (!env || !parts || !opts || !w0) return fail(GCNSA_ERR_ARG, "NULL argument");
  if (opts->n_layers < 1 || opts->n_layers > GCNSA_MAX_LAYERS) return fail(GCNSA_ERR_ARG, "n_layers out of range");
  for (int l = 0; l <= opts->n_layers; ++l)
    if (opts->dims[l] < 1) return fail(GCNSA_ERR_ARG, "layer width < 1");
  if (opts->dims[0] != parts->f || opts->dims[opts->n_layers] != parts->c)
    return fail(GCNSA_ERR_ARG, "dims[0] must equal f and dims[L] must equal c of the partitions");
  if (opts->gemm_mode != GCNSA_GEMM_FP32 && opts->gemm_mode != GCNSA_GEMM_TF32X3 && opts->gemm_mode != GCNSA_GEMM_TF32)
    return fail(GCNSA_ERR_ARG, "unknown gemm_mode");
  if (opts->agg_mode != GCNSA_AGG_GRAD_AVG && opts->agg_mode != GCNSA_AGG_PARAM_AVG)
    return fail(GCNSA_ERR_ARG, "unknown agg_mode");
  if (!(opts->lr > 0.f) || !(opts->beta1 >= 0.f && opts->beta1 < 1.f) || !(opts->beta2 >= 0.f && opts->beta2 < 1.f) ||
      !(opts->eps > 0.f))
    return fail(GCNSA_ERR_ARG, "Adam hyper-parameters out of range");
  int rc = check_device(env);
  if (rc) return rc;
  gcnsa_model* M = new (std::nothrow) gcnsa_model();
  if (!M) return fail(GCNSA_ERR_OOM, "host allocation failed");
  M->env.e = *env;
  M->o = *opts;
  M->L = opts->n_layers;
  M->m = parts->m;
  M->n_max = std::max<int64_t>(parts->n_max, 1);
  int64_t off = 0;
  M->ld_max = 0;
  for (int l = 0; l < M->L; ++l) {
    const int64_t din = opts->dims[l], dout = opts->dims[l + 1];
    M->w_ld[l] = GCNSA_LD(dout);
    M->w_off[l] = off; off += (din * M->w_ld[l] + 63) / 64 * 64;
    M->b_off[l] = off; off += (M->w_ld[l] + 63) / 64 * 64;
    M->transform_first[l] = dout <= din;  // multiply by W first when the layer does not widen
    if (l == 0 && opts->cache_ax) M->transform_first[l] = false;  // (A_hat X) W with A_hat X kept across epochs
    M->ld_max = std::max<int64_t>(M->ld_max, std::max<int64_t>(GCNSA_LD(din), GCNSA_LD(dout)));
  }
  M->count = off;
  auto fail_free = [&](int code) {
    std::string keep = g_err;
    gcnsa_model_destroy(M);
    g_err = keep;
    return code;
  };
  const size_t pbytes = (size_t)off * sizeof(float);
  M->theta = (float*)M->dalloc(pbytes); M->gsum = (float*)M->dalloc(pbytes);
  M->am = (float*)M->dalloc(pbytes);    M->av = (float*)M->dalloc(pbytes);
  const size_t act = (size_t)M->n_max * (size_t)M->ld_max * sizeof(float);
  M->loss_parts = (float*)M->dalloc((size_t)(M->m + 1) * sizeof(float));
  M->adam_state = (double*)M->dalloc(4 * sizeof(double));
  bool ok = M->theta && M->gsum && M->am && M->av && M->loss_parts && M->adam_state;
  if (ok && pbytes * (size_t)M->m <= kGradBytes) ok = (M->gparts = (float*)M->dalloc(pbytes * (size_t)M->m)) != nullptr;
  size_t ws = 0, sc = 0;
  for (int l = 0; l < M->L; ++l) {
    const int64_t din = opts->dims[l], dout = opts->dims[l + 1];
    // (partitions have at most n_max rows, and one with fewer may be cut into more slices)
    ws = std::max(ws, gemm_workspace_upto(opts->gemm_mode, 1, 0, din, dout, M->n_max, true));
    ws = std::max(ws, gemm_workspace_upto(opts->gemm_mode, 0, 0, M->n_max, dout, din, false));
    ws = std::max(ws, gemm_workspace_upto(opts->gemm_mode, 0, 1, M->n_max, din, dout, false));
    sc = std::max(sc, colsum_scratch(M->n_max, (int32_t)dout));
    sc = std::max(sc, gemm_colsum_scratch(M->n_max, (int32_t)din));  // the fused bias gradient of the layer below
    sc = std::max(sc, (size_t)4 * 148 * (size_t)((din + 3) / 4 * 4) * sizeof(float));  // ... as a narrow product leaves it
  }
  M->ws_bytes = ws; M->sc_bytes = sc;
  if (opts->factored_norm)
    for (const DevPart& d : parts->parts)
      for (int l = 0; l < M->L; ++l)
        M->dw_bytes = std::max(M->dw_bytes, spmm_planned_workspace(d.plan, std::min(opts->dims[l], opts->dims[l + 1])));
  M->lanes.resize(1);
  size_t lane_bytes = M->dw_bytes;
  ok = ok && alloc_lane(M, M->lanes[0], act, &lane_bytes);
  if (ok && opts->cache_ax) {
    M->ax.assign((size_t)parts->m, nullptr);
    M->ax_version.assign((size_t)parts->m, 0);
    M->ax_uid = parts->uid;
    for (int32_t p = 0; p < parts->m && ok; ++p) {
      const size_t bytes = (size_t)std::max<int64_t>(parts->parts[p].info.n, 1) * (size_t)parts->ldx * sizeof(float);
      M->ax[p] = (float*)M->dalloc(bytes);
      ok = M->ax[p] != nullptr;
      if (ok) cudaMemsetAsync(M->ax[p], 0, bytes, M->env.stream());
    }
  }
  if (ok && opts->agg_mode == GCNSA_AGG_PARAM_AVG) {
    const size_t pb = (size_t)M->count * sizeof(float);
    M->am_parts = (float*)M->dalloc(pb * M->m);
    M->av_parts = (float*)M->dalloc(pb * M->m);
    M->theta_acc = (float*)M->dalloc(pb);
    ok = M->am_parts && M->av_parts && M->theta_acc;
    if (ok) {
      cudaMemsetAsync(M->am_parts, 0, pb * M->m, M->env.stream());
      cudaMemsetAsync(M->av_parts, 0, pb * M->m, M->env.stream());
      cudaMemsetAsync(M->theta_acc, 0, pb, M->env.stream());
    }
  }
  if (!ok) return fail_free(fail(GCNSA_ERR_OOM, "device allocation failed"));
  // from here on what a model can do without: the workspace of the planned products (without it the products are gathers),
  // and the lanes after the first, which only make a recorded epoch faster
  if (M->dw_bytes && !(M->lanes[0].dw = M->dalloc(M->dw_bytes))) M->dw_bytes = 0;
  M->lanes.resize((size_t)epoch_lanes(M, parts, lane_bytes));
  if (M->gparts && beside(parts)) M->beside = std::min(parts->m, 3);
  for (size_t i = 1; i < M->lanes.size(); ++i) {
    const size_t mark = M->owned.size();
    Lane& W = M->lanes[i];
    if (alloc_lane(M, W, act) && (!M->dw_bytes || (W.dw = M->dalloc(M->dw_bytes)))) continue;
    while (M->owned.size() > mark) {
      M->env.release(M->owned.back());
      M->owned.pop_back();
    }
    M->lanes.resize(i);
  }
  cudaStream_t s = M->env.stream();
  cudaError_t e = cudaMemsetAsync(M->theta, 0, pbytes, s);
  if (e == cudaSuccess) e = cudaMemsetAsync(M->gsum, 0, pbytes, s);
  if (e == cudaSuccess) e = cudaMemsetAsync(M->am, 0, pbytes, s);
  if (e == cudaSuccess) e = cudaMemsetAsync(M->av, 0, pbytes, s);
  if (e == cudaSuccess && M->gparts) e = cudaMemsetAsync(M->gparts, 0, pbytes * (size_t)M->m, s);
  if (e == cudaSuccess) e = cudaMemsetAsync(M->loss_parts, 0, (size_t)(M->m + 1) * sizeof(float), s);
  if (e == cudaSuccess) e = cudaMemsetAsync(M->adam_state, 0, 4 * sizeof(double), s);
  for (Lane& W : M->lanes) {
    if (e == cudaSuccess) e = cudaMemsetAsync(W.tmp_a, 0, act, s);
    if (e == cudaSuccess) e = cudaMemsetAsync(W.tmp_b, 0, act, s);
    if (e == cudaSuccess && W.dw) e = cudaMemsetAsync(W.dw, 0, kPlannedHead, s);
    if (e == cudaSuccess) e = cudaMemsetAsync(W.dlogits, 0, (size_t)M->n_max * GCNSA_LD(parts->c) * sizeof(float), s);
    for (int l = 0; l < M->L && e == cudaSuccess; ++l) {
      e = cudaMemsetAsync(W.H[l + 1], 0, (size_t)M->n_max * GCNSA_LD(opts->dims[l + 1]) * sizeof(float), s);
      if (e == cudaSuccess && W.S[l])
        e = cudaMemsetAsync(W.S[l], 0, (size_t)M->n_max * GCNSA_LD(opts->dims[l]) * sizeof(float), s);
    }
  }
  if (e != cudaSuccess) return fail_free(cuda_fail(e, "cudaMemsetAsync"));
  for (int l = 0; l < M->L; ++l) {
    if (!w0[l]) return fail_free(fail(GCNSA_ERR_ARG, "w0[l] is NULL"));
    rc = copy_param(M, M->theta, l, true, (void*)w0[l], (size_t)opts->dims[l] * opts->dims[l + 1] * sizeof(float), false);
    if (rc == GCNSA_OK && b0 && b0[l])
      rc = copy_param(M, M->theta, l, false, (void*)b0[l], (size_t)opts->dims[l + 1] * sizeof(float), false);
    if (rc) return fail_free(rc);
  }
  *out = M;
  return GCNSA_OK;
}

// Y = epi(A_hat X) or, transposed, epi(A_hat^T X) on partition d.  use: all rows and columns, the rows that carry loss
// only, or only the columns that carry loss (X has zero rows elsewhere).  src_scaled: the rows of X have been
// multiplied by d^-1/2 already (factored_norm), so the pattern of A + I is all the product needs besides a row scale.
// With factored_norm a partition's plan takes the product where it has one; without it the stored values are read.
static int sparse_product(gcnsa_model* M, Lane& W, void* s, const DevPart& d, DenseUse use, bool transposed, bool src_scaled,
                          const float* x, int64_t ldx, int32_t f, int epi, const float* aux, int64_t ldaux, float* y,
                          int64_t ldy) {
  const int64_t n = d.info.n;
  const bool fact = M->o.factored_norm != 0;
  const int64_t rows = use == DenseUse::lossRows ? d.info.n_train : n;
  const int64_t nnz = use == DenseUse::lossRows ? d.m_nnz : use == DenseUse::lossCols ? d.tm_nnz : d.info.nnz;
  const bool values = !(fact && src_scaled);
  const SpmmCost cost = spmm_cost(rows, use == DenseUse::lossCols ? d.info.n_train : n, nnz, f, values, epi == GCNSA_EPI_MASK);
  const int32_t* rowptr = use == DenseUse::lossCols ? d.tm_rowptr : transposed ? d.t_rowptr : d.rowptr;
  const int32_t* col = use == DenseUse::lossCols ? d.tm_col : transposed ? d.t_col : d.col;
  // (gcnsa_evaluate may bring partitions the workspace was not sized for)
  if (fact && d.plan.n_chunks > 0 && spmm_planned_workspace(d.plan, f) <= M->dw_bytes) {
    M->prof_begin();
    const int r = launch_spmm_planned(s, d.plan, use, rows, rowptr, col, d.dinv, src_scaled ? nullptr : d.dinv, x, ldx, f, epi,
                                      aux, ldaux, y, ldy, W.dw, SpmmBounds{n, n, use == DenseUse::lossCols ? d.tm_nnz : d.info.nnz});
    if (r > 0) return cuda_fail((cudaError_t)r, "launch_spmm_planned");
    if (r == 0) {
      const int64_t rest = d.info.nnz ? (int64_t)((double)d.plan.r_nnz * (double)nnz / (double)d.info.nnz) : 0;
      const double mask_bytes = epi == GCNSA_EPI_MASK ? 4.0 * (double)f * (double)rows : 0.0;
      M->prof_end(0, cost.bytes, cost.flops, spmm_planned_l1_bytes(d.plan, use, rows, rest, f) + mask_bytes, cost.bytes_val);
      return GCNSA_OK;
    }
  }
  const int32_t* order = use == DenseUse::lossRows ? d.m_order : use == DenseUse::lossCols ? d.tm_order : transposed ? d.t_order : d.order;
  const int64_t n_long = use == DenseUse::lossRows ? d.m_n_long : use == DenseUse::lossCols ? d.tm_n_long : transposed ? d.t_n_long : d.n_long;
  const float* val = !values ? nullptr : use == DenseUse::lossCols ? d.tm_val : transposed ? d.t_val : d.val;
  PROF_SPMM(M, cost, launch_spmm(s, rows, rowptr, col, val, values ? nullptr : d.dinv, order, n_long, x, ldx, f, epi, aux, ldaux,
                                 y, ldy, SpmmBounds{n, n, use == DenseUse::lossCols ? d.tm_nnz : d.info.nnz},
                                 use == DenseUse::lossRows ? d.m_split : use == DenseUse::lossCols ? d.tm_split : transposed ? d.t_split : d.split));
  return GCNSA_OK;
}

// cache_ax: (re)computes A_hat X of partition p if its feature rows changed since the cached product was made
static int ensure_ax(gcnsa_model* M, const gcnsa_parts* P, int32_t p) {
  if (M->ax_version[p] == P->x_version[p]) return GCNSA_OK;
  const DevPart& d = P->parts[p];
  const int rc = sparse_product(M, M->lanes[0], M->env.e.stream, d, DenseUse::all, false, false, d.x, P->ldx, M->o.dims[0],
                                GCNSA_EPI_NONE, nullptr, 0, M->ax[p], P->ldx);
  if (rc) return rc;
  M->ax_version[p] = P->x_version[p];
  return GCNSA_OK;
}

static int check_model(const gcnsa_model* M, const gcnsa_parts* P) {
  if (P->m != M->m || P->f != M->o.dims[0] || P->c != M->o.dims[M->L] || P->n_max > M->n_max)
    return fail(GCNSA_ERR_ARG, "model was created for other partitions");
  return GCNSA_OK;
}

// The branches of an epoch that is being recorded.  There is one stream; a branch is the set of recorded nodes that its next
// launch depends on, and `use` makes that of another branch the stream's.  (A stream and events for each branch cost a first
// epoch 0.1 to 0.2 ms a branch, and a replay has the branches in its graph anyway.)
struct Fork {
  struct Deps {
    std::vector<cudaGraphNode_t> nodes;
    std::vector<cudaGraphEdgeData> edges;
    void add(const Deps& d) {
      for (size_t i = 0; i < d.nodes.size(); ++i)
        if (std::find(nodes.begin(), nodes.end(), d.nodes[i]) == nodes.end()) {
          nodes.push_back(d.nodes[i]);
          edges.push_back(d.edges[i]);
        }
    }
  };
  cudaStream_t s = nullptr;
  std::vector<Deps> at;
  int cur = 0;
  cudaError_t now(Deps* d) const {
    cudaStreamCaptureStatus status;
    const cudaGraphNode_t* nodes = nullptr;
    const cudaGraphEdgeData* edges = nullptr;
    size_t n = 0;
    const cudaError_t rc = cudaStreamGetCaptureInfo_v3(s, &status, nullptr, nullptr, &nodes, &edges, &n);
    if (rc != cudaSuccess) return rc;
    if (status != cudaStreamCaptureStatusActive) return cudaErrorStreamCaptureInvalidated;
    d->nodes.assign(nodes, nodes + n);
    if (edges) d->edges.assign(edges, edges + n);
    else d->edges.assign(n, cudaGraphEdgeData{});
    return cudaSuccess;
  }
  cudaError_t put(Deps& d) const {
    return cudaStreamUpdateCaptureDependencies_v2(s, d.nodes.data(), d.edges.data(), d.nodes.size(), cudaStreamSetCaptureDependencies);
  }
  // branches 0 (what the stream has been given so far) to n - 1
  void begin(cudaStream_t stream, int n) {
    s = stream;
    at.assign((size_t)n, Deps());
    cur = 0;
  }
  // what follows on the stream is branch k's
  cudaError_t use(int k) {
    if (k == cur) return cudaSuccess;
    cudaError_t rc = now(&at[cur]);
    if (rc == cudaSuccess) rc = put(at[k]);
    if (rc == cudaSuccess) cur = k;
    return rc;
  }
  // what branch k has been given so far
  cudaError_t mark(int k, Deps* d) const {
    if (k == cur) return now(d);
    *d = at[k];
    return cudaSuccess;
  }
  // branch k waits for what is in d
  cudaError_t wait(int k, const Deps& d) {
    if (k != cur) {
      at[k].add(d);
      return cudaSuccess;
    }
    Deps mine;
    cudaError_t rc = now(&mine);
    mine.add(d);
    return rc == cudaSuccess ? put(mine) : rc;
  }
  cudaError_t edge(int from, int to) {
    Deps d;
    const cudaError_t rc = mark(from, &d);
    return rc == cudaSuccess ? wait(to, d) : rc;
  }
};

// Where a recorded epoch puts what the next kernel of a pass does not read (the loss, bias gradients, the weight gradients
// of all layers but the first): a branch `side` beside the pass's branch `lane`.  fork == NULL: everything in a row.
struct Branch {
  Fork* fork = nullptr;
  int lane = 0, side = 0;
  // launches go to the branch, after what the pass has been given so far (also = false: after what it was given when it was
  // last asked), until back()
  cudaError_t aside(bool also = true) const {
    if (!fork) return cudaSuccess;
    const cudaError_t rc = also ? fork->edge(lane, side) : cudaSuccess;
    return rc == cudaSuccess ? fork->use(side) : rc;
  }
  cudaError_t back() const { return fork ? fork->use(lane) : cudaSuccess; }
};

// forward pass of partition p in the buffers of lane W on stream s; the partition's loss goes to loss_parts[p]
static int forward_lane(gcnsa_model* M, const gcnsa_parts* P, int32_t p, Lane& W, void* s, const Branch& br = Branch{}) {
  const DevPart& d = P->parts[p];
  const int64_t n = d.info.n;
  const float* h = d.x;
  int64_t ldh = P->ldx;
  const bool fact = M->o.factored_norm != 0;
  for (int l = 0; l < M->L; ++l) {
    const int32_t din = M->o.dims[l], dout = M->o.dims[l + 1];
    const bool last = l == M->L - 1;
    const float* bias = M->o.use_bias ? M->theta + M->b_off[l] : nullptr;
    const int epi = last ? (bias ? GCNSA_EPI_BIAS : GCNSA_EPI_NONE) : GCNSA_EPI_BIAS_RELU;
    const float* w = M->theta + M->w_off[l];
    const int64_t ldo = GCNSA_LD(dout);
    if (M->transform_first[l]) {
      // factored_norm: A_hat T = diag(dinv) (A + I) (diag(dinv) T): the GEMM's epilogue scales the rows of T and
      // the product reads no values
      if (narrow_ok(M->o.gemm_mode, n, dout, din, l == 0)) {
        NarrowArgs na;
        na.m = n; na.n = dout; na.k = din;
        na.a = h; na.lda = ldh;
        na.w = w; na.ldw = M->w_ld[l];
        na.w_ready = l > 0;  // (the optimizer may be the kernel before the first)
        na.c = W.tmp_a; na.ldc = ldo;
        na.row_scale = fact ? d.dinv : nullptr;
        PROF(M, 1, gemm_bytes(n, dout, din), 2.0 * n * dout * din, launch_narrow(s, na));
      } else {
        PROF(M, 1, gemm_bytes(n, dout, din), 2.0 * n * dout * din,
             launch_gemm(s, M->o.gemm_mode, 0, 0, n, dout, din, h, ldh, w, M->w_ld[l], W.tmp_a, ldo, 0,
                         fact ? GCNSA_EPI_ROWSCALE : GCNSA_EPI_NONE, fact ? d.dinv : nullptr, 0, W.ws, M->ws_bytes, M->beside));
      }
      // training reads the logits of the rows that carry loss only: the other rows are not computed
      const DenseUse use = last && M->o.loss_rows_only && !M->all_rows_once ? DenseUse::lossRows : DenseUse::all;
      const int rc = sparse_product(M, W, s, d, use, false, fact, W.tmp_a, ldo, dout, epi, bias, 0, W.H[l + 1], ldo);
      if (rc) return rc;
    } else {
      const float* agg = W.S[l];
      if (l == 0 && M->o.cache_ax && P->uid == M->ax_uid) {
        // A_hat X does not change between epochs: computed when the feature rows were (re)written, reused otherwise
        int rc = ensure_ax(M, P, p);
        if (rc) return rc;
        agg = M->ax[p];
      } else {
        const int rc = sparse_product(M, W, s, d, DenseUse::all, false, false, h, ldh, din, GCNSA_EPI_NONE, nullptr, 0, W.S[l], ldh);
        if (rc) return rc;
      }
      if (l == 0) W.s0_used = agg;
      PROF(M, 1, gemm_bytes(n, dout, din), 2.0 * n * dout * din,
           launch_gemm(s, M->o.gemm_mode, 0, 0, n, dout, din, agg, ldh, w, M->w_ld[l], W.H[l + 1], ldo, 0, epi, bias,
                       0, W.ws, M->ws_bytes, M->beside));
    }
    h = W.H[l + 1];
    ldh = ldo;
  }
  const int64_t ldc = GCNSA_LD(P->c);
  // the backward pass wants the column sums of the logit gradient (a bias) and, with factored_norm and a last layer that
  // multiplies by W first, diag(dinv) times it in tmp_a (free by now): made while the gradient is in registers
  CeSide side;
  if (ce_by_groups(P->c)) {
    if (M->o.use_bias) side.sums = W.ce_sums;
    if (fact && M->transform_first[M->L - 1]) {
      side.row_scale = d.dinv;
      side.scaled = W.tmp_a;
      side.lds = ldc;
    }
  }
  PROF(M, 2, (side.scaled ? 12.0 : 8.0) * n * P->c + 5.0 * n, 0.0,
       launch_softmax_ce(s, n, P->c, h, ldc, d.y, d.mask, d.info.n_train, br.fork ? nullptr : M->loss_parts + p, W.dlogits, ldc,
                         W.ce_part, side));
  if (br.fork) {
    CK(br.aside());
    CKL(launch_ce_loss(s, n, P->c, d.info.n_train, W.ce_part, M->loss_parts + p));
    CK(br.back());
  }
  return GCNSA_OK;
}

// backward pass of partition p after forward_lane in the same lane; dW, db go to grad (flat parameter layout), added
// to what is there when acc is 1
static int backward_lane(gcnsa_model* M, const gcnsa_parts* P, int32_t p, Lane& W, void* s, float* grad, int acc,
                         const Branch& br = Branch{}) {
  const DevPart& d = P->parts[p];
  const int64_t n = d.info.n;
  Fork::Deps q_read, sums_read;  // the branch's readers of tmp_b and of sc
  auto wait = [&](Fork::Deps& e) {
    const cudaError_t rc = e.nodes.empty() ? cudaSuccess : br.fork->wait(br.lane, e);
    e = Fork::Deps();
    return rc;
  };
  const float* g = W.dlogits;  // gradient w.r.t. Z^l, [n x LD(dims[l+1])]
  const bool fact = M->o.factored_norm != 0;
  bool bias_done = false, g_scaled = false;  // what the producer of g has done for this layer already
  for (int l = M->L - 1; l >= 0; --l) {
    const int32_t din = M->o.dims[l], dout = M->o.dims[l + 1];
    const int64_t ldo = GCNSA_LD(dout), ldi = GCNSA_LD(din);
    const float* hprev = l == 0 ? d.x : W.H[l];
    const float* w = M->theta + M->w_off[l];
    float* gw = grad + M->w_off[l];
    // with factored_norm the products of the layers that multiply by W first read diag(dinv) G: the column-sum
    // kernel, which reads every element of G anyway, writes that copy to tmp_a (G itself below the last layer)
    bool scaled = false;
    if (bias_done) {  // the masked product of the layer above has added the column sums (and scaled g) already
      scaled = g_scaled;
    } else if (l == M->L - 1 && ce_by_groups(dout)) {  // the softmax kernel has made the partial sums and the scaled copy
      scaled = fact && M->transform_first[l];
      if (M->o.use_bias) {
        CK(br.aside(false));
        PROF(M, 2, 0.0, 0.0, launch_ce_sums(s, n, dout, W.ce_sums, grad + M->b_off[l], acc));
        CK(br.back());
      }
    } else if (M->o.use_bias) {
      CK(wait(sums_read));
      if (fact && M->transform_first[l]) {
        PROF(M, 2, 12.0 * n * dout, 0.0,
             launch_colsum_scaled(s, n, dout, g, ldo, grad + M->b_off[l], acc, W.sc, d.dinv, W.tmp_a, ldo));
        scaled = true;
      } else {
        PROF(M, 2, 4.0 * n * dout, 0.0, launch_colsum(s, n, dout, g, ldo, grad + M->b_off[l], acc, W.sc));
      }
    }
    CK(wait(q_read));
    if (M->transform_first[l]) {
      // Q = A_hat^T G;  dW += H^{l-1}^T Q;  G^{l-1} = (Q W^T) .* [H^{l-1} > 0]
      if (fact) {
        // A_hat^T G = diag(dinv) (A + I)^T (diag(dinv) G): the scaled copy is in tmp_a (free at this point; for
        // the layers below the last, G is tmp_a itself and was scaled in place after its column sums were taken)
        if (!scaled) PROF(M, 2, 8.0 * n * dout, 0.0, launch_scale_rows(s, n, dout, d.dinv, g, ldo, W.tmp_a, ldo));
        g = W.tmp_a;
      }
      // the logit gradient has zero rows outside T_p: only the non-zeros whose column carries loss contribute
      const int rc = sparse_product(M, W, s, d, l == M->L - 1 ? DenseUse::lossCols : DenseUse::all, true, fact, g, ldo, dout,
                                    GCNSA_EPI_NONE, nullptr, 0, W.tmp_b, ldo);
      if (rc) return rc;
      // (the workspace has room for one of the two products of Q)
      const bool aside = br.fork && l > 0 && gemm_workspace(M->o.gemm_mode, 0, 1, n, din, dout) == 0;
      if (aside) CK(br.aside());
      PROF(M, 1, gemm_bytes(din, dout, n), 2.0 * n * dout * din,
           launch_gemm(s, M->o.gemm_mode, 1, 0, din, dout, n, hprev, ldi, W.tmp_b, ldo, gw, M->w_ld[l], acc,
                       GCNSA_EPI_NONE, nullptr, 0, W.ws, M->ws_bytes, M->beside));
      if (aside) {
        CK(br.fork->mark(br.side, &q_read));
        CK(br.back());
      }
      bias_done = g_scaled = false;
      if (l > 0 && M->o.use_bias) {
        // G^{l-1}, its column sums (the bias gradient of layer l - 1) and, where the next transposed product wants
        // it, diag(dinv) G^{l-1} in place: one pass in the product's epilogue
        const bool want_scaled = fact && M->transform_first[l - 1];
        int64_t left = 0;
        CK(wait(sums_read));
        if (narrow_ok(M->o.gemm_mode, n, din, dout, false)) {
          NarrowArgs na;
          na.m = n; na.n = din; na.k = dout;
          na.a = W.tmp_b; na.lda = ldo;
          na.w = w; na.ldw = M->w_ld[l]; na.w_t = true; na.w_ready = true;
          na.c = W.tmp_a; na.ldc = ldi;
          na.row_scale = want_scaled ? d.dinv : nullptr;
          na.mask = hprev; na.ldmask = ldi;
          na.sums = (float*)W.sc;
          PROF(M, 1, gemm_bytes(n, din, dout) + 4.0 * n * din, 2.0 * n * dout * din, launch_narrow(s, na));
          CK(br.aside());
          PROF(M, 1, 0.0, 0.0, launch_sum_rows(s, narrow_blocks(n, din), din, na.sums, (din + 3) / 4 * 4, grad + M->b_off[l - 1], acc,
                                               nullptr));
          if (br.fork) CK(br.fork->mark(br.side, &sums_read));
          CK(br.back());
        } else {
          PROF(M, 1, gemm_bytes(n, din, dout) + 4.0 * n * din, 2.0 * n * dout * din,
               launch_gemm_mask_colsum(s, M->o.gemm_mode, 0, 1, n, din, dout, W.tmp_b, ldo, w, M->w_ld[l], W.tmp_a, ldi, hprev,
                                       ldi, want_scaled ? d.dinv : nullptr, grad + M->b_off[l - 1], acc, W.sc, W.ws,
                                       M->ws_bytes, br.fork ? &left : nullptr));
          if (left) {
            CK(br.aside());
            CKL(launch_mask_colsum_rest(s, left, n, din, grad + M->b_off[l - 1], acc, W.sc));
            CK(br.fork->mark(br.side, &sums_read));
            CK(br.back());
          }
        }
        bias_done = true;
        g_scaled = want_scaled;
        g = W.tmp_a;
      } else if (l > 0) {
        PROF(M, 1, gemm_bytes(n, din, dout) + 4.0 * n * din, 2.0 * n * dout * din,
             launch_gemm(s, M->o.gemm_mode, 0, 1, n, din, dout, W.tmp_b, ldo, w, M->w_ld[l], W.tmp_a, ldi, 0, GCNSA_EPI_MASK,
                         hprev, ldi, W.ws, M->ws_bytes, M->beside));
        g = W.tmp_a;
      }
    } else {
      bias_done = g_scaled = false;
      // dW += S^T G;  R = G W^T;  G^{l-1} = (A_hat^T R) .* [H^{l-1} > 0]
      PROF(M, 1, gemm_bytes(din, dout, n), 2.0 * n * dout * din,
           launch_gemm(s, M->o.gemm_mode, 1, 0, din, dout, n, l == 0 ? W.s0_used : W.S[l], ldi, g, ldo, gw, M->w_ld[l], acc,
                       GCNSA_EPI_NONE, nullptr, 0, W.ws, M->ws_bytes, M->beside));
      if (l > 0) {
        PROF(M, 1, gemm_bytes(n, din, dout), 2.0 * n * dout * din,
             launch_gemm(s, M->o.gemm_mode, 0, 1, n, din, dout, g, ldo, w, M->w_ld[l], W.tmp_b, ldi, 0,
                         fact ? GCNSA_EPI_ROWSCALE : GCNSA_EPI_NONE, fact ? d.dinv : nullptr, 0, W.ws, M->ws_bytes, M->beside));
        // (on the last layer R = G W^T has the zero rows of G)
        const int rc = sparse_product(M, W, s, d, l == M->L - 1 ? DenseUse::lossCols : DenseUse::all, true, fact, W.tmp_b, ldi,
                                      din, GCNSA_EPI_MASK, hprev, ldi, W.tmp_a, ldi);
        if (rc) return rc;
        g = W.tmp_a;
      }
    }
  }
  if (br.fork) CK(br.fork->edge(br.side, br.lane));
  return GCNSA_OK;
}

int gcnsa_forward(gcnsa_model* M, const gcnsa_parts* P, int32_t p, float* loss_dev) {
  if (!M || !P || p < 0 || p >= P->m) return fail(GCNSA_ERR_ARG, "bad partition index or NULL");
  int rc = check_model(M, P);
  if (rc) return rc;
  rc = forward_lane(M, P, p, M->lanes[0], M->env.e.stream);
  if (rc) return rc;
  if (loss_dev)
    CK(cudaMemcpyAsync(loss_dev, M->loss_parts + p, sizeof(float), cudaMemcpyDeviceToDevice, M->env.stream()));
  M->last_forward = p;
  M->last_n = P->parts[p].info.n;
  return GCNSA_OK;
}

int gcnsa_backward(gcnsa_model* M, const gcnsa_parts* P, int32_t p) {
  if (!M || !P || p < 0 || p >= P->m) return fail(GCNSA_ERR_ARG, "bad partition index or NULL");
  if (M->last_forward != p) return fail(GCNSA_ERR_ORDER, "gcnsa_backward needs gcnsa_forward on the same partition first");
  if (M->accumulated >= M->m) return fail(GCNSA_ERR_ORDER, "all M partitions are accumulated already: call gcnsa_step");
  void* s = M->env.e.stream;
  const int rc = backward_lane(M, P, p, M->lanes[0], s, M->gsum, 1);
  if (rc) return rc;
  if (M->o.agg_mode == GCNSA_AGG_PARAM_AVG) {
    // this partition's own optimizer step from the aggregated parameters (Section 3.2), folded into the mean
    if (M->accumulated == 0)  // t -> t + 1 once per epoch
      PROF(M, 2, 0.0, 0.0, launch_adam_advance(s, M->adam_state, M->o.beta1, M->o.beta2));
    PROF(M, 2, 32.0 * M->count, 0.0,
         launch_adam_local_dev(s, M->count, M->theta, M->gsum, M->am_parts + (size_t)p * M->count,
                               M->av_parts + (size_t)p * M->count, M->theta_acc, M->accumulated == 0,
                               1.0f / (float)M->m, M->o.lr, M->o.beta1, M->o.beta2, M->o.eps, M->adam_state));
  }
  M->last_forward = -1;
  M->accumulated += 1;
  return GCNSA_OK;
}

int gcnsa_step(gcnsa_model* M) {
  if (!M) return fail(GCNSA_ERR_ARG, "model is NULL");
  if (M->accumulated != M->m) return fail(GCNSA_ERR_ORDER, "gcnsa_step needs one backward pass per partition");
  M->t += 1;
  if (M->o.agg_mode == GCNSA_AGG_PARAM_AVG) {
    CK(cudaMemcpyAsync(M->theta, M->theta_acc, (size_t)M->count * sizeof(float), cudaMemcpyDeviceToDevice, M->env.stream()));
    M->accumulated = 0;
    return GCNSA_OK;
  }
  PROF(M, 2, 0.0, 0.0, launch_adam_advance(M->env.e.stream, M->adam_state, M->o.beta1, M->o.beta2));  // t -> t + 1
  PROF(M, 2, 28.0 * M->count, 0.0,
       launch_adam_dev(M->env.e.stream, M->count, M->theta, M->gsum, M->am, M->av, 1.0f / (float)M->m, M->o.lr,
                       M->o.beta1, M->o.beta2, M->o.eps, M->adam_state));
  M->accumulated = 0;
  return GCNSA_OK;
}

// forward and backward pass of partition p of an epoch in lane W (without buffers of their own, as the calls step by step)
static int epoch_partition(gcnsa_model* M, const gcnsa_parts* P, int32_t p, Lane& W, cudaStream_t s, const Branch& br = Branch{}) {
  if (!M->gparts) {
    const int rc = gcnsa_forward(M, P, p, nullptr);
    return rc ? rc : gcnsa_backward(M, P, p);
  }
  const int rc = forward_lane(M, P, p, W, s, br);
  return rc ? rc : backward_lane(M, P, p, W, s, M->gparts + (size_t)p * M->count, 0, br);
}

// the step from the gradients of all partitions in gparts, on top of what gcnsa_model_set has left in the gradient sum;
// advanced: the step count has been advanced already.  (Not before the passes of plain launches: where one fails, the count
// on the device stays that of the host.)
static int optimizer_step(gcnsa_model* M, cudaStream_t s, bool advanced) {
  if (!M->gparts) return gcnsa_step(M);
  if (!advanced) PROF(M, 2, 0.0, 0.0, launch_adam_advance(s, M->adam_state, M->o.beta1, M->o.beta2));  // t -> t + 1
  const float inv_m = 1.0f / (float)M->m;
  if (M->o.agg_mode == GCNSA_AGG_PARAM_AVG)
    PROF(M, 2, 32.0 * M->count * M->m, 0.0,
         launch_adam_local_parts(s, M->count, M->m, M->theta, M->gsum, M->gparts, M->am_parts, M->av_parts, inv_m, M->o.lr,
                                 M->o.beta1, M->o.beta2, M->o.eps, M->adam_state));
  else
    PROF(M, 2, (24.0 + 4.0 * M->m) * M->count, 0.0,
         launch_adam_parts(s, M->count, M->m, M->theta, M->gsum, M->gparts, M->am, M->av, inv_m, M->o.lr, M->o.beta1, M->o.beta2,
                           M->o.eps, M->adam_state));
  M->t += 1;
  return GCNSA_OK;
}

// One epoch: forward and backward of every partition, each with a gradient buffer of its own (see kGradBytes), then the
// optimizer over all of them.  fork == NULL: everything on the model's stream, partition after partition.  Otherwise lane i takes
// partitions ..., i counted from the last one backwards in steps of the number of lanes (so lane 0 ends with the
// activations of the last partition, as without lanes) on a branch of its own; the sums are added in partition order
// in both cases, so the results are the same bit for bit.
static int epoch_body(gcnsa_model* M, const gcnsa_parts* P, float* loss_dev, Fork* fork) {
  int rc = check_model(M, P);
  if (rc) return rc;
  cudaStream_t s = M->env.stream();
  // branches: the lanes, one for the step count and the loss, one beside every lane
  const int lanes = fork ? (int)M->lanes.size() : 1, aux = lanes;
  if (fork) {
    fork->begin(s, 2 * lanes + 1);
    for (int i = 1; i <= lanes; ++i) CK(fork->edge(0, i));
  }
  const bool early = fork && M->gparts;  // (beside the passes)
  if (early) {
    CK(fork->use(aux));
    PROF(M, 2, 0.0, 0.0, launch_adam_advance(s, M->adam_state, M->o.beta1, M->o.beta2));  // t -> t + 1
  }
  for (int32_t p = 0; p < P->m; ++p) {
    const int lane = (P->m - 1 - p) % lanes;
    Branch br;
    if (early && branches(P)) br = Branch{fork, lane, lanes + 1 + lane};
    if (fork) CK(fork->use(lane));
    rc = epoch_partition(M, P, p, M->lanes[lane], s, br);
    if (rc) return rc;
  }
  if (fork) {
    CK(fork->use(0));
    for (int i = 1; i <= lanes; ++i) CK(fork->edge(i, 0));
  }
  if (loss_dev) {
    if (fork) {
      CK(fork->edge(0, aux));
      CK(fork->use(aux));
    }
    CKL(launch_mean(s, M->loss_parts, M->m, loss_dev));
    if (fork) CK(fork->use(0));
  }
  rc = optimizer_step(M, s, early);
  if (rc) return rc;
  if (loss_dev && fork) CK(fork->edge(aux, 0));
  M->last_forward = -1;
  M->last_n = P->parts[P->m - 1].info.n;
  return GCNSA_OK;
}

int gcnsa_epoch(gcnsa_model* M, const gcnsa_parts* P, float* loss_dev) {
  if (!M || !P) return fail(GCNSA_ERR_ARG, "NULL argument");
  if (M->accumulated != 0) return fail(GCNSA_ERR_ORDER, "gcnsa_epoch needs an empty gradient sum");
  cudaStream_t s = M->env.stream();
  const bool want_graph = M->o.epoch_graph && !M->graph_off && !M->prof_on && s != nullptr;
  if (!want_graph) return epoch_body(M, P, loss_dev, nullptr);
  if (M->o.cache_ax && P->uid == M->ax_uid && P->m == M->m)  // outside the recording: a replay only reads the cached products
    for (int32_t p = 0; p < P->m; ++p) {
      int rc = ensure_ax(M, P, p);
      if (rc) return rc;
    }
  if (M->graph_exec && (M->graph_parts_uid != P->uid || M->graph_loss != (const void*)loss_dev)) {
    cudaGraphExecDestroy(M->graph_exec);
    M->graph_exec = nullptr;
  }
  if (!M->graph_exec) {
    // record one epoch; the launches only describe work, nothing runs until the graph is launched
    const int64_t t0 = M->t;
    const int64_t launches0 = gcnsa_launch_count();
    cudaGraph_t graph = nullptr;
    int rc = GCNSA_OK;
    Fork fork;
    if (cudaStreamBeginCapture(s, cudaStreamCaptureModeThreadLocal) != cudaSuccess) {
      cudaGetLastError();
      M->graph_off = true;
      return epoch_body(M, P, loss_dev, nullptr);
    }
    rc = epoch_body(M, P, loss_dev, &fork);
    cudaError_t e = cudaStreamEndCapture(s, &graph);
    M->t = t0;  // the host's copy of the step count advances when the graph runs
    M->accumulated = 0;
    M->last_forward = -1;
    const int recorded = (int)(gcnsa_launch_count() - launches0);
    note_launch(-recorded);  // recorded, not launched
    if (rc != GCNSA_OK || e != cudaSuccess || !graph ||
        cudaGraphInstantiate(&M->graph_exec, graph, 0) != cudaSuccess) {
      if (graph) cudaGraphDestroy(graph);
      cudaGetLastError();
      M->graph_exec = nullptr;
      M->graph_off = true;  // this stream or driver cannot record the epoch: plain launches from now on
      return epoch_body(M, P, loss_dev, nullptr);
    }
    cudaGraphDestroy(graph);
    M->graph_parts_uid = P->uid;
    M->graph_loss = (const void*)loss_dev;
    M->graph_kernels = recorded;
  }
  CK(cudaGraphLaunch(M->graph_exec, s));
  note_launch(M->graph_kernels);
  M->last_forward = -1;  // its activations are gone
  M->t += 1;
  M->last_n = P->parts[P->m - 1].info.n;
  return GCNSA_OK;
}

int gcnsa_epoch_host(gcnsa_model* M, gcnsa_parts* P, const float* const* x_host, float* loss_host) {
  if (!M || !P || !x_host || !loss_host) return fail(GCNSA_ERR_ARG, "NULL argument");
  if (M->accumulated != 0) return fail(GCNSA_ERR_ORDER, "gcnsa_epoch_host needs an empty gradient sum");
  for (int32_t p = 0; p < P->m; ++p)
    if (!x_host[p]) return fail(GCNSA_ERR_ARG, "x_host[p] is NULL");
  int rc = check_model(M, P);
  if (rc) return rc;
  cudaStream_t s = M->env.stream();
  if (!P->copy_stream) {  // first use: copy stream, events, two staging buffers
    CK(cudaStreamCreateWithFlags(&P->copy_stream, cudaStreamNonBlocking));
    P->ready.resize((size_t)P->m);
    for (int32_t p = 0; p < P->m; ++p) CK(cudaEventCreateWithFlags(&P->ready[p], cudaEventDisableTiming));
    P->consumed.resize(2);
    for (cudaEvent_t& e : P->consumed) {
      CK(cudaEventCreateWithFlags(&e, cudaEventDisableTiming));
      CK(cudaEventRecord(e, s));
    }
  }
  for (int b = 0; b < 2; ++b) {  // (a call that ran out of memory here leaves what it got for the next one)
    if (P->staging[b]) continue;
    P->staging[b] = (float*)P->dalloc((size_t)std::max<int64_t>(P->n_max, 1) * (size_t)P->f * sizeof(float));
    if (!P->staging[b]) return fail(GCNSA_ERR_OOM, "device allocation failed");
  }
  // Uploads run back to back on their own stream, two staging buffers ahead of the compute stream, which spreads the dense
  // rows over the padded device rows itself: on the copy stream that kernel stood between two copies (58 241 x 602 in four
  // partitions: 45 us each).  The epoch takes the copies (2.8 ms at 50 GB/s) and the last partition's passes: 3.45 -> 3.28 ms.
  auto copy_in = [&](int32_t p) {
    cudaError_t e = cudaStreamWaitEvent(P->copy_stream, P->consumed[p & 1], 0);  // the buffer's previous rows have been read
    if (e == cudaSuccess)
      e = cudaMemcpyAsync(P->staging[p & 1], x_host[p], (size_t)P->parts[p].info.n * (size_t)P->f * sizeof(float),
                          cudaMemcpyHostToDevice, P->copy_stream);
    return e == cudaSuccess ? cudaEventRecord(P->ready[p], P->copy_stream) : e;
  };
  auto epoch = [&]() -> int {
    for (int32_t p = 0; p < std::min(P->m, 2); ++p) CK(copy_in(p));
    for (int32_t p = 0; p < P->m; ++p) {
      const DevPart& d = P->parts[p];
      CK(cudaStreamWaitEvent(s, P->ready[p], 0));
      CKL(launch_copy_rows(s, d.info.n, P->f, P->staging[p & 1], P->f, d.x, P->ldx));
      P->x_version[p] += 1;
      CK(cudaEventRecord(P->consumed[p & 1], s));
      if (p + 2 < P->m) CK(copy_in(p + 2));
      const int r = epoch_partition(M, P, p, M->lanes[0], s);
      if (r) return r;
    }
    return optimizer_step(M, s, false);
  };
  rc = epoch();
  if (rc) {  // copies may be on their way: the caller's buffers are not read after the call
    cudaStreamSynchronize(P->copy_stream);
    return rc;
  }
  M->last_forward = -1;
  M->last_n = P->parts[P->m - 1].info.n;
  float* mean_dev = M->loss_parts + M->m;  // slot after the M partition losses
  CKL(launch_mean(M->env.e.stream, M->loss_parts, M->m, mean_dev));
  CK(cudaMemcpyAsync(loss_host, mean_dev, sizeof(float), cudaMemcpyDeviceToHost, M->env.stream()));
  CK(cudaStreamSynchronize(M->env.stream()));
  return GCNSA_OK;
}

}  // extern "C"

// ------------------------------------------------------- get / set / ops ---
extern "C" {

static float* param_base(const gcnsa_model* M, int32_t what, bool* is_w) {
  switch (what) {
    case GCNSA_GET_W: *is_w = true; return M->theta;
    case GCNSA_GET_B: *is_w = false; return M->theta;
    case GCNSA_GET_GRAD_W: *is_w = true; return M->gsum;
    case GCNSA_GET_GRAD_B: *is_w = false; return M->gsum;
    case GCNSA_GET_ADAM_M_W: *is_w = true; return M->am_parts ? M->am_parts + (size_t)M->state_p * M->count : M->am;
    case GCNSA_GET_ADAM_M_B: *is_w = false; return M->am_parts ? M->am_parts + (size_t)M->state_p * M->count : M->am;
    case GCNSA_GET_ADAM_V_W: *is_w = true; return M->av_parts ? M->av_parts + (size_t)M->state_p * M->count : M->av;
    case GCNSA_GET_ADAM_V_B: *is_w = false; return M->av_parts ? M->av_parts + (size_t)M->state_p * M->count : M->av;
    default: return nullptr;
  }
}

int gcnsa_model_get(const gcnsa_model* M, int32_t what, int32_t layer, void* host_dst, size_t bytes) {
  if (!M || !host_dst) return fail(GCNSA_ERR_ARG, "NULL argument");
  bool is_w = false;
  if (float* base = param_base(M, what, &is_w)) {
    if (layer < 0 || layer >= M->L) return fail(GCNSA_ERR_ARG, "layer out of range");
    return copy_param(M, base, layer, is_w, host_dst, bytes, true);
  }
  const float* src = nullptr;
  int64_t cols = 0;
  if (what == GCNSA_GET_ACT) {
    if (layer < 1 || layer > M->L) return fail(GCNSA_ERR_ARG, "layer out of range");
    src = M->lanes[0].H[layer];
    cols = M->o.dims[layer];
  } else if (what == GCNSA_GET_DLOGITS) {
    src = M->lanes[0].dlogits;
    cols = M->o.dims[M->L];
  } else {
    return fail(GCNSA_ERR_ARG, "unknown tensor id");
  }
  if (bytes != (size_t)(M->last_n * cols) * sizeof(float)) return fail(GCNSA_ERR_ARG, "byte count does not match the tensor");
  if (M->last_n > 0 && cols > 0) {
    // A strided copy to the host goes row by row (rows of 80 bytes: 21 GB/s), a dense one at 55 GB/s: rows without padding
    // are one piece, others are packed on the device first (tmp_b: no pass leaves anything there).  An evaluation that
    // fetches the logits: 116 483 x 41 1 595 -> 1 336 us, 20 000 x 20 201 -> 162, x 41 246 -> 209, x 5 165 -> 160.
    if (GCNSA_LD(cols) != cols) {
      std::lock_guard<std::mutex> lock(M->pack);
      CKL(launch_copy_rows(M->env.e.stream, M->last_n, cols, src, GCNSA_LD(cols), M->lanes[0].tmp_b, cols));
      CK(cudaMemcpyAsync(host_dst, M->lanes[0].tmp_b, bytes, cudaMemcpyDeviceToHost, M->env.stream()));
    } else {
      CK(cudaMemcpyAsync(host_dst, src, bytes, cudaMemcpyDeviceToHost, M->env.stream()));
    }
  }
  CK(cudaStreamSynchronize(M->env.stream()));
  return GCNSA_OK;
}

int gcnsa_model_set(gcnsa_model* M, int32_t what, int32_t layer, const void* host_src, size_t bytes) {
  if (!M || !host_src) return fail(GCNSA_ERR_ARG, "NULL argument");
  bool is_w = false;
  float* base = param_base(M, what, &is_w);
  if (!base) return fail(GCNSA_ERR_ARG, "tensor cannot be set");
  if (layer < 0 || layer >= M->L) return fail(GCNSA_ERR_ARG, "layer out of range");
  return copy_param(M, base, layer, is_w, (void*)host_src, bytes, false);
}

int gcnsa_model_profile(gcnsa_model* M, int32_t enable) {
  if (!M) return fail(GCNSA_ERR_ARG, "model is NULL");
  CK(cudaStreamSynchronize(M->env.stream()));
  M->prof_on = enable != 0;
  M->recs.clear();
  return GCNSA_OK;
}

int gcnsa_model_profile_read(gcnsa_model* M, gcnsa_profile* out) {
  if (!M || !out) return fail(GCNSA_ERR_ARG, "NULL argument");
  std::memset(out, 0, sizeof(*out));
  CK(cudaStreamSynchronize(M->env.stream()));
  for (size_t i = 0; i < M->recs.size(); ++i) {
    float ms = 0.f;
    CK(cudaEventElapsedTime(&ms, M->ev[2 * i], M->ev[2 * i + 1]));
    const auto& r = M->recs[i];
    out->ms[r.cat] += ms;
    out->launches[r.cat] += r.launches;
    out->alg_bytes[r.cat] += r.bytes;
    out->l1_bytes[r.cat] += r.l1;
    out->alg_bytes_val[r.cat] += r.bytes_val;
    out->flops[r.cat] += r.flops;
  }
  M->recs.clear();
  return GCNSA_OK;
}

int gcnsa_evaluate(gcnsa_model* M, const gcnsa_parts* P, int32_t p, const uint8_t* mask_host, int64_t* correct_host,
                   int64_t* total_host, int32_t* pred_host) {
  if (!M || !P || !correct_host || !total_host || p < 0 || p >= P->m)
    return fail(GCNSA_ERR_ARG, "bad partition index or NULL");
  if (M->accumulated != 0 || M->last_forward >= 0)
    return fail(GCNSA_ERR_ORDER, "gcnsa_evaluate between a forward pass and gcnsa_step");
  if (!M->ev_pred) M->ev_pred = (int32_t*)M->dalloc((size_t)M->n_max * sizeof(int32_t));
  if (!M->ev_hits) M->ev_hits = (int32_t*)M->dalloc(4096 * sizeof(int32_t));
  if (!M->ev_mask) M->ev_mask = (uint8_t*)M->dalloc((size_t)M->n_max);
  if (!M->ev_pred || !M->ev_hits || !M->ev_mask) return fail(GCNSA_ERR_OOM, "device allocation failed");
  int rc = check_model(M, P);
  if (rc) return rc;
  const DevPart& d = P->parts[p];
  const int64_t n = d.info.n;
  cudaStream_t s = M->env.stream();
  // (before the forward pass: a copy from pageable memory holds the host up, and behind the pass the device would wait)
  if (mask_host && n > 0) CK(cudaMemcpyAsync(M->ev_mask, mask_host, (size_t)n, cudaMemcpyHostToDevice, s));
  M->all_rows_once = true;
  rc = gcnsa_forward(M, P, p, nullptr);
  M->all_rows_once = false;
  if (rc) return rc;
  M->last_forward = -1;                       // an evaluation pass is not followed by a backward pass
  int blocks = 0;
  CKL(launch_argmax_hits(s, n, P->c, M->lanes[0].H[M->L], GCNSA_LD(P->c), d.y, mask_host ? M->ev_mask : nullptr, M->ev_pred,
                         M->ev_hits, &blocks));
  std::vector<int32_t> hits((size_t)std::max(blocks, 1), 0);
  if (n > 0) CK(cudaMemcpyAsync(hits.data(), M->ev_hits, (size_t)blocks * sizeof(int32_t), cudaMemcpyDeviceToHost, s));
  if (pred_host && n > 0) CK(cudaMemcpyAsync(pred_host, M->ev_pred, (size_t)n * sizeof(int32_t), cudaMemcpyDeviceToHost, s));
  CK(cudaStreamSynchronize(s));
  int64_t correct = 0, total = 0;
  for (int b = 0; b < blocks && n > 0; ++b) correct += hits[b];
  for (int64_t i = 0; i < n; ++i) total += mask_host ? (mask_host[i] != 0) : 1;
  *correct_host = correct;
  *total_host = total;
  return GCNSA_OK;
}

int gcnsa_model_copy_params(gcnsa_model* dst, const gcnsa_model* src) {
  if (!dst || !src) return fail(GCNSA_ERR_ARG, "NULL argument");
  if (dst->L != src->L || dst->count != src->count) return fail(GCNSA_ERR_ARG, "models have different dims");
  for (int l = 0; l <= dst->L; ++l)
    if (dst->o.dims[l] != src->o.dims[l]) return fail(GCNSA_ERR_ARG, "models have different dims");
  CK(cudaStreamSynchronize(src->env.stream()));
  CK(cudaMemcpyAsync(dst->theta, src->theta, (size_t)dst->count * sizeof(float), cudaMemcpyDeviceToDevice,
                     dst->env.stream()));
  return GCNSA_OK;
}

int gcnsa_model_select_partition(gcnsa_model* M, int32_t p) {
  if (!M || p < 0 || p >= M->m) return fail(GCNSA_ERR_ARG, "NULL model or partition index out of range");
  M->state_p = p;
  return GCNSA_OK;
}

int gcnsa_model_get_t(const gcnsa_model* M, int64_t* t_out) {
  if (!M || !t_out) return fail(GCNSA_ERR_ARG, "NULL argument");
  *t_out = M->t;
  return GCNSA_OK;
}
int gcnsa_model_set_t(gcnsa_model* M, int64_t t) {
  if (!M || t < 0) return fail(GCNSA_ERR_ARG, "NULL model or negative step count");
  M->t = t;
  // the kernels read the count from device memory; the bias corrections are recomputed at the next step
  const double state[4] = {(double)t, 0.0, 0.0, 0.0};
  CK(cudaMemcpyAsync(M->adam_state, state, sizeof(state), cudaMemcpyHostToDevice, M->env.stream()));
  CK(cudaStreamSynchronize(M->env.stream()));
  return GCNSA_OK;
}

static bool aligned16(const void* p) { return ((uintptr_t)p & 15) == 0; }

int gcnsa_op_spmm(void* stream, int64_t n_rows, const int32_t* rowptr, const int32_t* col, const float* val,
                  const int32_t* order, int64_t n_long, const float* x, int64_t ldx, int32_t f, int32_t epi, const float* aux,
                  int64_t ldaux, float* y, int64_t ldy) {
  if (n_rows < 0 || f < 0 || n_rows >= INT32_MAX) return fail(GCNSA_ERR_ARG, "negative or oversized dimension");
  if (n_rows == 0 || f == 0) return GCNSA_OK;
  if (!rowptr || !col || !val || !x || !y) return fail(GCNSA_ERR_ARG, "NULL pointer");
  if (ldx % 4 || ldy % 4 || ldx < f || ldy < f || !aligned16(x) || !aligned16(y))
    return fail(GCNSA_ERR_ARG, "x and y need 16-byte aligned bases and leading dimensions that are multiples of 4");
  if (epi < GCNSA_EPI_NONE || epi > GCNSA_EPI_MASK) return fail(GCNSA_ERR_ARG, "unknown epilogue");
  if (epi == GCNSA_EPI_MASK && (!aux || ldaux % 4 || ldaux < f || !aligned16(aux)))
    return fail(GCNSA_ERR_ARG, "mask needs a 16-byte aligned base and a leading dimension that is a multiple of 4");
  if (epi == GCNSA_EPI_BIAS && !aux) return fail(GCNSA_ERR_ARG, "bias is NULL");
  if (n_long < 0 || n_long > n_rows) return fail(GCNSA_ERR_ARG, "n_long out of range");
  CKL(launch_spmm(stream, n_rows, rowptr, col, val, nullptr, order, n_long, x, ldx, f, epi, aux, ldaux, y, ldy,
                  SpmmBounds{n_rows, -1, -1}));
  return GCNSA_OK;
}

int gcnsa_op_spmm_pattern(void* stream, int64_t n_rows, const int32_t* rowptr, const int32_t* col, const float* row_scale,
                          const int32_t* order, int64_t n_long, const float* x, int64_t ldx, int32_t f, int32_t epi,
                          const float* aux, int64_t ldaux, float* y, int64_t ldy) {
  if (n_rows < 0 || f < 0 || n_rows >= INT32_MAX) return fail(GCNSA_ERR_ARG, "negative or oversized dimension");
  if (n_rows == 0 || f == 0) return GCNSA_OK;
  if (!rowptr || !col || !x || !y) return fail(GCNSA_ERR_ARG, "NULL pointer");
  if (ldx % 4 || ldy % 4 || ldx < f || ldy < f || !aligned16(x) || !aligned16(y))
    return fail(GCNSA_ERR_ARG, "x and y need 16-byte aligned bases and leading dimensions that are multiples of 4");
  if (epi < GCNSA_EPI_NONE || epi > GCNSA_EPI_MASK) return fail(GCNSA_ERR_ARG, "unknown epilogue");
  if (epi == GCNSA_EPI_MASK && (!aux || ldaux % 4 || ldaux < f || !aligned16(aux)))
    return fail(GCNSA_ERR_ARG, "mask needs a 16-byte aligned base and a leading dimension that is a multiple of 4");
  if (epi == GCNSA_EPI_BIAS && !aux) return fail(GCNSA_ERR_ARG, "bias is NULL");
  if (n_long < 0 || n_long > n_rows) return fail(GCNSA_ERR_ARG, "n_long out of range");
  CKL(launch_spmm(stream, n_rows, rowptr, col, nullptr, row_scale, order, n_long, x, ldx, f, epi, aux, ldaux, y, ldy,
                  SpmmBounds{n_rows, -1, -1}));
  return GCNSA_OK;
}

size_t gcnsa_op_gemm_workspace(int32_t mode, int32_t ta, int32_t tb, int64_t m, int64_t n, int64_t k) {
  if (m <= 0 || n <= 0 || k <= 0) return 0;
  return gemm_workspace(mode, ta, tb, m, n, k);
}

int gcnsa_tc_status(int32_t* status_host) {
  if (!status_host) return fail(GCNSA_ERR_ARG, "NULL argument");
  CK(cudaDeviceSynchronize());
  int v = 0;
  CKL(tc_status(&v));
  *status_host = v;
  return GCNSA_OK;
}

int gcnsa_debug_status(int32_t* enabled_host, int32_t* code_host, int64_t* value_host) {
  if (!enabled_host || !code_host || !value_host) return fail(GCNSA_ERR_ARG, "NULL argument");
#ifdef GCNSA_DEBUG
  *enabled_host = 1;
#else
  *enabled_host = 0;
#endif
  *code_host = 0;
  *value_host = 0;
  CK(cudaDeviceSynchronize());
  unsigned long long w[3] = {0ull, 0ull, 0ull};
  CKL(debug_word_spmm(&w[0], true));
  CKL(debug_word_build(&w[1], true));
  CKL(debug_word_dense(&w[2], true));
  const unsigned long long first = w[0] ? w[0] : w[1] ? w[1] : w[2];
  *code_host = (int32_t)(first >> 56);
  *value_host = (int64_t)(first & 0x00ffffffffffffffull);
  return GCNSA_OK;
}

int gcnsa_tc_clear(void) {
  CK(cudaDeviceSynchronize());
  CKL(tc_clear());
  return GCNSA_OK;
}

int gcnsa_op_gemm(void* stream, int32_t mode, int32_t ta, int32_t tb, int64_t m, int64_t n, int64_t k, const float* a,
                  int64_t lda, const float* b, int64_t ldb, float* c, int64_t ldc, int32_t accumulate, int32_t epi,
                  const float* aux, int64_t ldaux, void* workspace, size_t workspace_bytes) {
  if (m < 0 || n < 0 || k < 0) return fail(GCNSA_ERR_ARG, "negative dimension");
  if (mode != GCNSA_GEMM_FP32 && mode != GCNSA_GEMM_TF32X3 && mode != GCNSA_GEMM_TF32)
    return fail(GCNSA_ERR_ARG, "unknown gemm mode");
  if (m == 0 || n == 0) return GCNSA_OK;
  if (!c || (k > 0 && (!a || !b))) return fail(GCNSA_ERR_ARG, "NULL pointer");
  if (lda < (ta ? m : k) || ldb < (tb ? k : n) || ldc < n) return fail(GCNSA_ERR_ARG, "leading dimension too small");
  if (epi < GCNSA_EPI_NONE || epi > GCNSA_EPI_ROWSCALE) return fail(GCNSA_ERR_ARG, "unknown epilogue");
  if ((epi == GCNSA_EPI_MASK || epi == GCNSA_EPI_BIAS || epi == GCNSA_EPI_ROWSCALE) && !aux)
    return fail(GCNSA_ERR_ARG, "aux is NULL");
  CKL(launch_gemm(stream, mode, ta, tb, m, n, k, a, lda, b, ldb, c, ldc, accumulate, epi, aux, ldaux, workspace,
                  workspace_bytes));
  return GCNSA_OK;
}

size_t gcnsa_op_gemm_mask_colsum_scratch(int64_t m, int32_t n) {
  return (gemm_colsum_scratch(m < 0 ? 0 : m, n < 0 ? 0 : n) + 255) / 256 * 256;
}

int gcnsa_op_gemm_mask_colsum(void* stream, int32_t mode, int32_t ta, int32_t tb, int64_t m, int64_t n, int64_t k,
                              const float* a, int64_t lda, const float* b, int64_t ldb, float* c, int64_t ldc,
                              const float* mask, int64_t ldmask, const float* row_scale, float* out,
                              int32_t accumulate, void* scratch, size_t scratch_bytes, void* workspace,
                              size_t workspace_bytes) {
  if (m < 0 || n < 0 || k < 0 || n >= (1LL << 31)) return fail(GCNSA_ERR_ARG, "negative dimension");
  if (mode != GCNSA_GEMM_FP32 && mode != GCNSA_GEMM_TF32X3 && mode != GCNSA_GEMM_TF32)
    return fail(GCNSA_ERR_ARG, "unknown gemm mode");
  if (n > 0 && !out) return fail(GCNSA_ERR_ARG, "NULL pointer");
  if (m == 0 || n == 0) {
    CKL(launch_gemm_mask_colsum(stream, mode, ta, tb, m, n, k, a, lda, b, ldb, c, ldc, mask, ldmask, row_scale, out, accumulate,
                                scratch, workspace, workspace_bytes));
    return GCNSA_OK;
  }
  if (!c || !mask || (k > 0 && (!a || !b))) return fail(GCNSA_ERR_ARG, "NULL pointer");
  if (lda < (ta ? m : k) || ldb < (tb ? k : n) || ldc < n || ldmask < n) return fail(GCNSA_ERR_ARG, "leading dimension too small");
  if (!scratch || ((uintptr_t)scratch & 255) || scratch_bytes < gemm_colsum_scratch(m, (int32_t)n))
    return fail(GCNSA_ERR_ARG, "scratch missing, unaligned or too small");
  CKL(launch_gemm_mask_colsum(stream, mode, ta, tb, m, n, k, a, lda, b, ldb, c, ldc, mask, ldmask, row_scale, out, accumulate,
                              scratch, workspace, workspace_bytes));
  return GCNSA_OK;
}

static int probe_sms(int* sms) {
  int dev = 0;
  CK(cudaGetDevice(&dev));
  CK(cudaDeviceGetAttribute(sms, cudaDevAttrMultiProcessorCount, dev));
  return GCNSA_OK;
}

int gcnsa_op_gather_probe_warps(int32_t* warps_out) {
  if (!warps_out) return fail(GCNSA_ERR_ARG, "NULL pointer");
  int sms = 0;
  int rc = probe_sms(&sms);
  if (rc) return rc;
  *warps_out = gather_probe_warps(sms);
  return GCNSA_OK;
}

int gcnsa_op_gather_probe(void* stream, const float* x, int64_t ldx, int64_t n_rows, int32_t window_rows,
                          int32_t hit_every, int32_t rounds, float* out, size_t out_bytes) {
  if (!x || !out) return fail(GCNSA_ERR_ARG, "NULL pointer");
  if (ldx < 128 || (ldx % 4) || ((uintptr_t)x & 15) || ((uintptr_t)out & 15))
    return fail(GCNSA_ERR_ARG, "rows of at least 128 floats, 16-byte aligned");
  if (n_rows < 1 || n_rows >= (1LL << 31) || window_rows < 1 || window_rows > n_rows || hit_every < 0 || rounds < 0)
    return fail(GCNSA_ERR_ARG, "row counts, hit_every or rounds out of range");
  int sms = 0;
  int rc = probe_sms(&sms);
  if (rc) return rc;
  if (out_bytes < (size_t)gather_probe_warps(sms) * 128 * sizeof(float)) return fail(GCNSA_ERR_ARG, "out too small");
  CKL(launch_gather_probe(stream, x, ldx, n_rows, window_rows, hit_every, rounds, out, sms));
  return GCNSA_OK;
}

size_t gcnsa_op_softmax_ce_scratch(int64_t n) { return softmax_ce_scratch(n < 0 ? 0 : n); }

int gcnsa_op_softmax_ce(void* stream, int64_t n, int32_t c, const float* logits, int64_t ld, const int32_t* y,
                        const uint8_t* mask, int64_t n_train, float* loss_dev, float* grad, int64_t ldg, void* scratch,
                        size_t scratch_bytes) {
  if (n < 0 || c < 1 || n_train < 0) return fail(GCNSA_ERR_ARG, "negative dimension or c < 1");
  if (n > 0 && (!logits || !y || !mask || !grad)) return fail(GCNSA_ERR_ARG, "NULL pointer");
  if (ld < c || ldg < c) return fail(GCNSA_ERR_ARG, "leading dimension too small");
  if (!scratch || scratch_bytes < softmax_ce_scratch(n)) return fail(GCNSA_ERR_ARG, "scratch too small");
  CKL(launch_softmax_ce(stream, n, c, logits, ld, y, mask, n_train, loss_dev, grad, ldg, scratch));
  return GCNSA_OK;
}

size_t gcnsa_op_colsum_scratch(int64_t n, int32_t f) { return colsum_scratch(n < 0 ? 0 : n, f < 0 ? 0 : f); }

int gcnsa_op_colsum(void* stream, int64_t n, int32_t f, const float* g, int64_t ldg, float* out, int32_t accumulate,
                    void* scratch, size_t scratch_bytes) {
  if (n < 0 || f < 0) return fail(GCNSA_ERR_ARG, "negative dimension");
  if (f == 0) return GCNSA_OK;
  if (!out || (n > 0 && !g) || ldg < f) return fail(GCNSA_ERR_ARG, "NULL pointer or leading dimension too small");
  if (!scratch || scratch_bytes < colsum_scratch(n, f)) return fail(GCNSA_ERR_ARG, "scratch too small");
  CKL(launch_colsum(stream, n, f, g, ldg, out, accumulate, scratch));
  return GCNSA_OK;
}

int gcnsa_op_colsum_scaled(void* stream, int64_t n, int32_t f, const float* g, int64_t ldg, float* out, int32_t accumulate,
                           void* scratch, size_t scratch_bytes, const float* row_scale, float* scaled, int64_t lds) {
  if (n < 0 || f < 0) return fail(GCNSA_ERR_ARG, "negative dimension");
  if (f == 0) return GCNSA_OK;
  if (!out || (n > 0 && !g) || ldg < f) return fail(GCNSA_ERR_ARG, "NULL pointer or leading dimension too small");
  if (!scratch || scratch_bytes < colsum_scratch(n, f)) return fail(GCNSA_ERR_ARG, "scratch too small");
  if (!row_scale || !scaled) return fail(GCNSA_ERR_ARG, "row_scale or scaled is NULL");
  if (lds % 4 || ldg % 4 || lds < (f + 3) / 4 * 4 || ldg < (f + 3) / 4 * 4 || !aligned16(scaled) || !aligned16(g))
    return fail(GCNSA_ERR_ARG, "g and scaled need 16-byte aligned bases and leading dimensions that are multiples of 4");
  CKL(launch_colsum_scaled(stream, n, f, g, ldg, out, accumulate, scratch, row_scale, scaled, lds));
  return GCNSA_OK;
}

int gcnsa_op_adam(void* stream, int64_t count, float* theta, float* gsum, float* m, float* v, float inv_m, float lr,
                  float beta1, float beta2, float eps, int64_t t) {
  if (count < 0 || t < 1) return fail(GCNSA_ERR_ARG, "negative count or t < 1");
  if (count > 0 && (!theta || !gsum || !m || !v)) return fail(GCNSA_ERR_ARG, "NULL pointer");
  CKL(launch_adam(stream, count, theta, gsum, m, v, inv_m, lr, beta1, beta2, eps, t));
  return GCNSA_OK;
}

int gcnsa_op_normalize(void* stream, int64_t n_rows, const int32_t* rowptr, const int32_t* col, const int32_t* deg,
                       float* val) {
  if (n_rows < 0) return fail(GCNSA_ERR_ARG, "negative dimension");
  if (n_rows > 0 && (!rowptr || !col || !deg || !val)) return fail(GCNSA_ERR_ARG, "NULL pointer");
  CKL(launch_normalize(stream, n_rows, rowptr, col, deg, val));
  return GCNSA_OK;
}

}  // extern "C"

// ------------------------------------------------------------------- plan ---
struct gcnsa_plan {
  HostBuild hb;
  int32_t m = 0;
};

extern "C" {

int gcnsa_plan_create(const gcnsa_graph* g, const gcnsa_part_opts* opts, gcnsa_plan** out) {
  if (!out) return fail(GCNSA_ERR_ARG, "out is NULL");
  *out = nullptr;
  if (!g || !opts) return fail(GCNSA_ERR_ARG, "NULL argument");
  gcnsa_plan* pl = new (std::nothrow) gcnsa_plan();
  if (!pl) return fail(GCNSA_ERR_OOM, "host allocation failed");
  int rc = build_host(g, opts, &pl->hb);
  if (rc) {
    delete pl;
    return rc;
  }
  pl->m = opts->m;
  *out = pl;
  return GCNSA_OK;
}

int gcnsa_plan_info(const gcnsa_plan* plan, int32_t p, gcnsa_part_info* out) {
  if (!plan || !out || p < 0 || p >= plan->m) return fail(GCNSA_ERR_ARG, "bad partition index or NULL");
  const HostPart& hp = plan->hb.parts[p];
  out->n_owned = hp.n_owned; out->n_halo = hp.n_halo; out->n = hp.n; out->nnz = hp.nnz; out->nts = hp.nts;
  out->n_train = hp.n_train; out->max_depth = hp.max_depth;
  return GCNSA_OK;
}

int gcnsa_plan_assignment(const gcnsa_plan* plan, int32_t* part_host) {
  if (!plan || !part_host) return fail(GCNSA_ERR_ARG, "NULL argument");
  std::memcpy(part_host, plan->hb.part.data(), plan->hb.part.size() * sizeof(int32_t));
  return GCNSA_OK;
}

int gcnsa_plan_export(const gcnsa_plan* plan, int32_t p, const gcnsa_part_host* dst) {
  if (!plan || !dst || p < 0 || p >= plan->m) return fail(GCNSA_ERR_ARG, "bad partition index or NULL");
  const HostPart& hp = plan->hb.parts[p];
  if (dst->rowptr) std::memcpy(dst->rowptr, hp.rowptr.data(), hp.rowptr.size() * sizeof(int32_t));
  if (dst->col) std::memcpy(dst->col, hp.col.data(), hp.col.size() * sizeof(int32_t));
  if (dst->t_rowptr) std::memcpy(dst->t_rowptr, hp.t_rowptr.data(), hp.t_rowptr.size() * sizeof(int32_t));
  if (dst->t_col) std::memcpy(dst->t_col, hp.t_col.data(), hp.t_col.size() * sizeof(int32_t));
  if (dst->members) std::memcpy(dst->members, hp.members.data(), hp.members.size() * sizeof(int64_t));
  if (dst->depth) std::memcpy(dst->depth, hp.depth.data(), hp.depth.size() * sizeof(int32_t));
  return GCNSA_OK;
}

int gcnsa_plan_export_schedule(const gcnsa_plan* plan, int32_t p, gcnsa_part_schedule_info* info,
                               const gcnsa_part_schedule_host* dst) {
  if (!plan || p < 0 || p >= plan->m) return fail(GCNSA_ERR_ARG, "bad partition index or NULL");
  const HostPart& hp = plan->hb.parts[p];
  if (info) {
    info->n_long = hp.n_long; info->t_n_long = hp.t_n_long; info->m_n_long = hp.m_n_long; info->tm_n_long = hp.tm_n_long;
    info->m_nnz = hp.m_nnz; info->tm_nnz = (int64_t)hp.tm_col.size();
  }
  if (!dst) return GCNSA_OK;
  auto put = [](int32_t* to, const std::vector<int32_t>& from) {
    if (to && !from.empty()) std::memcpy(to, from.data(), from.size() * sizeof(int32_t));
  };
  put(dst->order, hp.order); put(dst->t_order, hp.t_order); put(dst->m_order, hp.m_order);
  put(dst->tm_rowptr, hp.tm_rowptr); put(dst->tm_col, hp.tm_col); put(dst->tm_order, hp.tm_order);
  return GCNSA_OK;  // mask and y are gathered on the device only
}

int gcnsa_plan_destroy(gcnsa_plan* plan) {
  delete plan;
  return GCNSA_OK;
}

}  // extern "C"
