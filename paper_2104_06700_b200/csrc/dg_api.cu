// The C ABI of libdgagg: argument checks, handle bookkeeping and kernel dispatch.
// Declarations and the meaning of every argument are in include/dg.h.
#include <stdarg.h>
#include <stdio.h>
#include <stdlib.h>
#include <string.h>

#include <new>

#include "dg_internal.cuh"

namespace dg {

static thread_local char g_last_error[512] = "";
static std::atomic<int64_t> g_launches{0};

void set_error(const char* fmt, ...) {
  va_list ap;
  va_start(ap, fmt);
  vsnprintf(g_last_error, sizeof(g_last_error), fmt, ap);
  va_end(ap);
}

dg_status_t cuda_fail(cudaError_t e, const char* what) {
  set_error("%s: %s", what, cudaGetErrorString(e));
  return DG_ERR_CUDA;
}

void count_launches(int64_t k) { g_launches.fetch_add(k, std::memory_order_relaxed); }

static dg_status_t invalid(const char* msg) {
  set_error("%s", msg);
  return DG_ERR_INVALID_ARG;
}

// [a, a + a_bytes) and [b, b + b_bytes) share a byte
static bool overlaps(const void* a, size_t a_bytes, const void* b, size_t b_bytes) {
  const uintptr_t x = (uintptr_t)a, y = (uintptr_t)b;
  return x < y + b_bytes && y < x + a_bytes;
}

static inline size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }

// Returns everything a handle holds; kernels that still read it may be queued on any stream.
static void free_owned(Graph* g) {
  pool_retire(g->device, g->owned, g->owned_bytes);
  pool_retire(g->device, g->plan_memory, g->plan_bytes);
  pinned_counters_retire(g->device, g->host);
  if (g->col_totals_ready) cudaEventDestroy(g->col_totals_ready);
  for (size_t i = 0; i < g->aux_event_count; ++i) cudaEventDestroy(g->aux_events[i]);
  free(g->aux_events);
  if (g->aux_ready)
    for (int i = 0; i < 2; ++i) cudaStreamDestroy(g->aux_stream[i]);
  pool_close(g->device);
}

// Cost of a chunk (see Plan).  A large graph gets chunks of 1024: long enough to hide their start-up,
// short enough that a late one does not matter.  A smaller one is cut into kChunksPerSm chunks per SM, so
// that every SM has warps to hide latency with and the last wave is short, down to 64 entries, because
// more cut rows make the join dearer; and into chunks of 32 (one index batch) where there are at most
// kShortChunksPerSm of those (396 k edges, rows of 42, F = 64: 24.6 us at 32, 28.7 at 64; 619 k edges, rows up
// to 1400, F = 100: 76 / 69).  Measured, us
// of both directions with their joins at 32 / 64 / 128 / 256: 65 k edges, F = 64: 15 / 19 / 27 / 39;
// 1.2 M, F = 47: 72 / 66 / 67 / 74; 6.2 M, F = 100: 454 / 392 / 379 / 396; 16 M, F = 64 (columns up to
// 10^5 entries): 1286 / 1040 / 930 / 892.
// Rows up to twice a chunk stay whole: four times costs 2 to 15 % on the same graphs.  With the smallest
// chunks rows up to kFewEdgesRow entries do: such a call is short against its launches, and the join of
// cut rows is one more launch with scratch of its own, 4.5 us of host time and 3.5 us on the device (125 k
// edges, rows up to 157, forward + backward: 31.4 us cut at 64, 20.5 whole).  A compromise over graphs of 57 to 344 k
// edges: rows of 20 to 300, F = 4 20.5 us at 160, 13.8 at 512; rows to 700, F = 16 27.6 / 21.0, F = 256 65.9 / 73.9;
// power-law rows, F = 64 24.7 / 36.9; 300 rows of 100 to 1500, F = 64 26.9 / 32.4.
// Rows over kLongestWhole entries are cut whatever the caller's threshold: a whole row is one warp's chain of fp32
// additions (4 M entries, message add: relative error 1.4e-3 whole, 1.9e-7 in pieces; 2 M entries, F = 128: 197 and 1.3 ms).
constexpr int64_t kMaxChunk = 1024, kMinChunk = 32, kChunksPerSm = 320, kRowCost = 8;
constexpr int64_t kShortChunksPerSm = 108, kFewEdgesRow = 160, kLongestWhole = 4096;
static int64_t chunk_cost(const Graph* g) {
  const int64_t total = g->nnz + kRowCost * g->n;
  int64_t cost;
  if (g->rows_per_block > 0) {  // the caller's rows per warp, at the average row length
    cost = (g->rows_per_block + 7) / 8 * (g->nnz / (g->n > 0 ? g->n : 1) + kRowCost);
    cost = cost < 32 ? 32 : cost;
  } else {
    cost = total / (g->sm_count * kChunksPerSm);
    if (cost < 64) cost = total <= g->sm_count * kShortChunksPerSm * kMinChunk ? kMinChunk : 64;
    if (cost > kMaxChunk) cost = kMaxChunk;
  }
  return (cost + 31) & ~(int64_t)31;
}
// Cost of a row beside its entries; at least a 31st of a chunk, so that no chunk has more than 31 rows.
static int64_t row_cost(const Graph* g) {
  const int64_t least = (chunk_cost(g) + 30) / 31;
  return least > kRowCost ? least : kRowCost;
}
static int64_t cut_threshold(const Graph* g) {
  if (g->heavy_threshold > 0) return g->heavy_threshold < kLongestWhole ? g->heavy_threshold : kLongestWhole;
  return g->rows_per_block == 0 && chunk_cost(g) == kMinChunk ? kFewEdgesRow : 2 * chunk_cost(g);
}

// Where the totals of the rows' (0) or the columns' (1) plan lie among the counters.
static int totals_of(const Graph* g, int columns) { return kTotals + (2 * g->totals_set + columns) * kTotalsPerPlan; }

// Takes the memory of both plans for the current chunk cost and threshold; on failure the plans are as they were.
static dg_status_t reserve_plans(Graph* g) {
  const int64_t cost = chunk_cost(g);
  const int64_t count = (g->nnz + row_cost(g) * g->n + cost - 1) / cost;
  const int64_t cuts = g->nnz > cut_threshold(g) ? count : 0;
  const size_t chunk_bytes = align256((size_t)(count + 1) * sizeof(Chunk));
  const size_t cut_bytes = align256((size_t)cuts * sizeof(CutRow));
  const size_t bytes = 2 * (chunk_bytes + cut_bytes);
  void* memory = nullptr;
  DG_CUDA(pool_alloc(g->device, bytes, 0, &memory));
  g->plan_memory = memory;
  g->plan_bytes = bytes;
  char* p = static_cast<char*>(memory);
  Plan* both[2] = {&g->row_plan, &g->col_plan};
  for (int i = 0; i < 2; ++i) {
    Plan& plan = *both[i];
    plan.chunks = reinterpret_cast<Chunk*>(p);
    p += chunk_bytes;
    plan.cuts = reinterpret_cast<CutRow*>(p);
    p += cut_bytes;
    plan.totals = g->counters + totals_of(g, i);
    plan.count = count;
    plan.max_cuts = cuts;
    // a row of m > threshold entries holds at most m / cost + 1 boundaries
    plan.max_slots = cuts ? g->nnz / cost + g->nnz / cut_threshold(g) + 1 : 0;
    if (plan.max_slots > count) plan.max_slots = count;
    plan.slots = plan.cut_rows = plan.most_pieces = cuts ? -1 : 0;
  }
  return DG_OK;
}

static dg_status_t plan_rows(Graph* g, cudaStream_t s) {
  return build_plan(g->rowptr, g->n, g->nnz, chunk_cost(g), row_cost(g), cut_threshold(g), g->row_plan, s);
}

static void take_totals(const Graph* g, int columns, Plan* plan) {
  const int32_t* v = g->host->v + totals_of(g, columns);
  plan->slots = v[0];
  plan->cut_rows = v[1];
  plan->most_pieces = v[2];
}

// What follows every transposition: the columns' plan, its totals sent to the host behind it (read by
// the first backward pass that finds the copy finished; until then their bounds serve).
dg_status_t finish_transpose(Graph* g, cudaStream_t s) {
  if (dg_status_t st = build_plan(g->colptr, g->n, g->nnz, chunk_cost(g), row_cost(g), cut_threshold(g), g->col_plan,
                                     s))
    return st;
  if (g->col_plan.max_cuts == 0) return DG_OK;
  g->col_plan.slots = g->col_plan.cut_rows = g->col_plan.most_pieces = -1;
  const int at = totals_of(g, 1);
  DG_CUDA(cudaMemcpyAsync(g->host->v + at, g->counters + at, kTotalsPerPlan * sizeof(int32_t),
                          cudaMemcpyDeviceToHost, s));
  DG_CUDA(cudaEventRecord(g->col_totals_ready, s));
  return DG_OK;
}

const Plan& column_plan(Graph* g) {
  if (g->col_plan.slots < 0) {
    if (cudaEventQuery(g->col_totals_ready) == cudaSuccess) {
      take_totals(g, 1, &g->col_plan);
    } else {
      (void)cudaGetLastError();  // "not ready" must not be mistaken for a failed launch later
    }
  }
  return g->col_plan;
}

static dg_status_t build_plans(Graph* g) {
  if (dg_status_t st = plan_rows(g, 0)) return st;
  DG_CUDA(cudaMemcpyAsync(g->host, g->counters, sizeof(HostCounters), cudaMemcpyDeviceToHost, 0));
  if (g->transposed)
    if (dg_status_t st = finish_transpose(g, 0)) return st;
  DG_CUDA(cudaDeviceSynchronize());
  return DG_OK;
}

// Sets *knob, which the chunk cost or the cut threshold follows, and makes new plans.  The old ones may be in use,
// or being built, on any stream: waits for the device on both sides.  If that fails, knob and plans are as before.
static dg_status_t replan(Graph* g, int64_t* knob, int64_t value) {
  const DeviceScope scope(g->device);
  DG_CUDA(pool_wait(g->device));
  const Graph before = *g;
  *knob = value;
  g->totals_set ^= 1;
  dg_status_t st = reserve_plans(g);
  if (st == DG_OK) st = build_plans(g);
  if (st == DG_OK) {
    take_totals(g, 0, &g->row_plan);
    pool_retire(g->device, before.plan_memory, before.plan_bytes);
    return DG_OK;
  }
  if (g->plan_memory != before.plan_memory) pool_retire(g->device, g->plan_memory, g->plan_bytes);
  *g = before;
  return st;
}

static dg_status_t check_features(const Graph* g, const void* in, size_t in_elem_bytes, float* out,
                                  int32_t F, dg_op_t op) {
  if (!g) return invalid("graph handle is NULL");
  if (F < 1) return invalid("F must be >= 1");
  if (F > (1 << 20)) {
    set_error("F must be at most 2^20");
    return DG_ERR_UNSUPPORTED;
  }
  if (op != DG_OP_SUM && op != DG_OP_MEAN) return invalid("op must be DG_OP_SUM or DG_OP_MEAN");
  if (g->n > 0) {
    if (!in || !out) return invalid("feature matrix pointer is NULL");
    const size_t elems = (size_t)g->n * (size_t)F;
    const uintptr_t x = (uintptr_t)in, y = (uintptr_t)out;
    if (x < y + elems * sizeof(float) && y < x + elems * in_elem_bytes)
      return invalid("input and output feature matrices overlap");
  }
  return DG_OK;
}

// Forward / backward AP for either storage type of the gathered matrix.
// `loops`: implicit self loops in this call.
static dg_status_t run_forward(Graph* g, const void* H, bool bf16, int32_t F, dg_op_t op, bool loops,
                               float* out, void* stream) {
  if (dg_status_t st = check_features(g, H, bf16 ? 2 : 4, out, F, op)) return st;
  ApArgs a{};
  a.ptr = g->rowptr;
  a.idx = g->colidx;
  a.w = g->edge_w;
  a.X = H;
  a.x_bf16 = bf16;
  a.Y = out;
  a.n = g->n;
  a.F = F;
  a.mean_rows = op == DG_OP_MEAN;
  const SelfArgs sa{loops ? g->rowptr : nullptr, op == DG_OP_MEAN};
  return aggregate_run(g, a, sa, g->row_plan, g->split_csr, (cudaStream_t)stream);
}

static dg_status_t run_backward(Graph* g, const void* dOut, bool bf16, int32_t F, dg_op_t op, bool loops,
                                float* dH, void* stream) {
  if (dg_status_t st = check_features(g, dOut, bf16 ? 2 : 4, dH, F, op)) return st;
  if (!g->transposed) {
    set_error("the backward pass needs dg_graph_transpose first");
    return DG_ERR_NOT_TRANSPOSED;
  }
  if (op == DG_OP_MEAN && loops != (g->self_loops_in_csc != 0)) {
    set_error("the CSC was built with another value of self_loops: transpose again");
    return DG_ERR_NOT_TRANSPOSED;
  }
  ApArgs a{};
  a.ptr = g->colptr;
  a.idx = g->rowidx_T;
  a.w = op == DG_OP_MEAN ? g->mean_scale_T : g->w_T;
  a.mean_factors = op == DG_OP_MEAN && !g->edge_w;
  a.X = dOut;
  a.x_bf16 = bf16;
  a.Y = dH;
  a.n = g->n;
  a.F = F;
  a.mean_rows = 0;
  const SelfArgs sa{loops ? g->rowptr : nullptr, op == DG_OP_MEAN};
  return aggregate_run(g, a, sa, column_plan(g), g->split_csc, (cudaStream_t)stream);
}

// sum_k w_k X[idx[k]] over the CSR rows (or the CSC columns) with the sum / mean kernels, for
// the operator pairs of the general entry points that are exactly this.  w is in the order of
// the direction walked, or nullptr; the handle's own weights and its "self_loops" attribute play
// no part.
dg_status_t aggregate_sum(Graph* g, bool over_csc, const float* w, const float* X, int32_t F,
                          float* Y, cudaStream_t s) {
  ApArgs a{};
  a.ptr = over_csc ? g->colptr : g->rowptr;
  a.idx = over_csc ? g->rowidx_T : g->colidx;
  a.w = w;
  a.X = X;
  a.Y = Y;
  a.n = g->n;
  a.F = F;
  return aggregate_run(g, a, SelfArgs{nullptr, 0}, over_csc ? column_plan(g) : g->row_plan,
                       over_csc ? g->split_csc : g->split_csr, s);
}

static dg_status_t malformed(int flags) {
  set_error("malformed CSR:%s%s%s%s", (flags & 1) ? " rowptr[0] != 0;" : "",
            (flags & 2) ? " rowptr decreases;" : "", (flags & 4) ? " rowptr[n] != nnz;" : "",
            (flags & 8) ? " colidx outside [0, n);" : "");
  return DG_ERR_INVALID_GRAPH;
}

}  // namespace dg

using namespace dg;

extern "C" {

dg_status_t dg_graph_create(int64_t n, int64_t nnz, const int64_t* rowptr,
                            const int32_t* colidx, const float* edge_w, dg_graph_t* out_graph) {
  if (!out_graph) return invalid("out_graph is NULL");
  *out_graph = nullptr;
  if (n < 0 || nnz < 0) return invalid("n and nnz must be >= 0");
  if (n >= ((int64_t)1 << 31) || nnz >= ((int64_t)1 << 31)) {
    set_error("n and nnz must be below 2^31");
    return DG_ERR_UNSUPPORTED;
  }
  if (!rowptr) return invalid("rowptr is NULL");
  if (nnz > 0 && !colidx) return invalid("colidx is NULL");
  if (nnz > 0 && n == 0) return invalid("edges without vertices");

  Graph* g = new (std::nothrow) Graph();
  if (!g) return invalid("out of host memory");
  g->n = n;
  g->nnz = nnz;
  g->rowptr = rowptr;
  g->colidx = colidx;
  g->edge_w = edge_w;
  // attributes, not cudaGetDeviceProperties: that call alone took 2.6 ms
  int l2 = 0;
  cudaError_t e = cudaGetDevice(&g->device);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&g->sm_count, cudaDevAttrMultiProcessorCount, g->device);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&l2, cudaDevAttrL2CacheSize, g->device);
  if (e == cudaSuccess) e = pool_open(g->device);
  if (e != cudaSuccess) { delete g; return cuda_fail(e, "device query"); }
  g->l2_bytes = (size_t)l2;
  g->l2_budget_bytes = (int64_t)(g->l2_bytes * 3 / 8);  // 47 of 126 MB: see aggregate_run
  g->fine_rows = (n + kFineBlocks - 1) / kFineBlocks;
  if (g->fine_rows < 1) g->fine_rows = 1;

  // The caller may have produced the arrays on any stream: wait for the device once, then everything
  // below runs on the default stream and is waited for once, at the end.
  dg_status_t st = DG_OK;
  e = pool_wait(g->device);
  const bool split = wants_split(n, nnz);
  const size_t counter_bytes = align256(sizeof(HostCounters));
  const size_t split_bytes = split ? align256((size_t)(kFineBlocks + 1) * (size_t)n * sizeof(int32_t)) : 0;
  g->owned_bytes = counter_bytes + split_bytes;
  if (e == cudaSuccess) e = pool_alloc(g->device, g->owned_bytes, 0, &g->owned);
  if (e == cudaSuccess) e = pinned_counters(&g->host);
  if (e == cudaSuccess) e = cudaEventCreateWithFlags(&g->col_totals_ready, cudaEventDisableTiming);
  if (e == cudaSuccess) {
    char* p = static_cast<char*>(g->owned);
    g->counters = reinterpret_cast<int32_t*>(p);
    if (split) g->split_csr = reinterpret_cast<int32_t*>(p + counter_bytes);
    e = cudaMemsetAsync(g->counters, 0, sizeof(HostCounters), 0);
  }
  if (e != cudaSuccess) st = cuda_fail(e, "graph metadata");

  // The kernels gather X[colidx[k]] without a range check, so a malformed CSR must never reach
  // them: one streaming pass over rowptr and colidx here (about a millisecond per 10^9 edges).
  if (st == DG_OK) st = reserve_plans(g);
  if (st == DG_OK) st = check_csr(g, g->counters + kFlags, 0);
  if (st == DG_OK) st = plan_rows(g, 0);
  if (st == DG_OK && split)
    st = build_split(rowptr, colidx, n, g->fine_rows, g->split_csr, g->counters + kUnsorted,
                     g->counters + kFlags, 0);
  if (st == DG_OK) {
    e = cudaMemcpyAsync(g->host, g->counters, sizeof(HostCounters), cudaMemcpyDeviceToHost, 0);
    if (e == cudaSuccess) e = cudaStreamSynchronize(0);
    if (e != cudaSuccess) st = cuda_fail(e, "graph create");
  }
  if (st == DG_OK && g->host->v[kFlags]) st = malformed(g->host->v[kFlags]);
  if (st != DG_OK) { free_owned(g); delete g; return st; }
  take_totals(g, 0, &g->row_plan);
  if (g->host->v[kUnsorted]) g->split_csr = nullptr;  // rows not sorted: no source blocking
  *out_graph = g;
  return DG_OK;
}

dg_status_t dg_graph_destroy(dg_graph_t g) {
  if (!g) return DG_OK;
  free_owned(g);
  delete g;
  return DG_OK;
}

dg_status_t dg_graph_validate(dg_graph_t g, void* stream) {
  if (!g) return invalid("graph handle is NULL");
  cudaStream_t s = (cudaStream_t)stream;
  int32_t flags = 0;
  if (dg_status_t st = check_csr(g, g->counters + kFlags, s)) return st;
  DG_CUDA(cudaMemcpyAsync(&flags, g->counters + kFlags, sizeof(flags), cudaMemcpyDeviceToHost, s));
  DG_CUDA(cudaStreamSynchronize(s));
  return flags ? malformed(flags) : DG_OK;
}

dg_status_t dg_graph_transpose_workspace(dg_graph_t g, size_t* csc_bytes, size_t* scratch_bytes) {
  if (!g) return invalid("graph handle is NULL");
  if (!csc_bytes || !scratch_bytes) return invalid("size output is NULL");
  transpose_sizes(g->n, g->nnz, g->edge_w != nullptr, csc_bytes, scratch_bytes);
  return DG_OK;
}

dg_status_t dg_graph_transpose(dg_graph_t g, void* csc_storage, size_t csc_bytes, void* scratch,
                               size_t scratch_bytes, void* stream) {
  if (!g) return invalid("graph handle is NULL");
  if (!csc_storage || !scratch) return invalid("csc_storage or scratch is NULL");
  if (((uintptr_t)csc_storage | (uintptr_t)scratch) & 255)
    return invalid("csc_storage and scratch must be 256-byte aligned");
  size_t need_csc, need_scratch;
  transpose_sizes(g->n, g->nnz, g->edge_w != nullptr, &need_csc, &need_scratch);
  if (csc_bytes < need_csc || scratch_bytes < need_scratch) {
    set_error("workspace smaller than dg_graph_transpose_workspace reports");
    return DG_ERR_WORKSPACE;
  }
  if (overlaps(csc_storage, need_csc, scratch, need_scratch))
    return invalid("csc_storage and scratch overlap");
  g->transposed = false;
  if (dg_status_t st = transpose_run(g, csc_storage, scratch, (cudaStream_t)stream)) return st;
  g->transposed = true;
  return finish_transpose(g, (cudaStream_t)stream);
}

dg_status_t dg_graph_update_weights(dg_graph_t g, void* stream) {
  if (!g) return invalid("graph handle is NULL");
  if (!g->edge_w) return invalid("the graph has no edge weights");
  if (!g->transposed) return DG_OK;  // the CSR is read in place: nothing to refresh
  return refresh_csc_weights(g, (cudaStream_t)stream);
}

dg_status_t dg_graph_get_csc(dg_graph_t g, const int64_t** colptr, const int32_t** rowidx_T,
                             const float** w_T, const int32_t** perm) {
  if (!g) return invalid("graph handle is NULL");
  if (!g->transposed) {
    set_error("dg_graph_transpose has not been called");
    return DG_ERR_NOT_TRANSPOSED;
  }
  if (colptr) *colptr = g->colptr;
  if (rowidx_T) *rowidx_T = g->rowidx_T;
  if (w_T) *w_T = g->w_T;
  if (perm) *perm = g->perm;
  return DG_OK;
}

dg_status_t dg_aggregate_fwd(dg_graph_t g, const float* H, int32_t F, dg_op_t op, float* out,
                             void* stream) {
  return run_forward(g, H, false, F, op, g && g->self_loops, out, stream);
}

dg_status_t dg_aggregate_fwd_self(dg_graph_t g, const float* H, int32_t F, dg_op_t op, float* out,
                                  void* stream) {
  return run_forward(g, H, false, F, op, true, out, stream);
}

dg_status_t dg_aggregate_bwd_self(dg_graph_t g, const float* dOut, int32_t F, dg_op_t op, float* dH,
                                  void* stream) {
  return run_backward(g, dOut, false, F, op, true, dH, stream);
}

dg_status_t dg_layer_fwd(dg_graph_t g, float* Y, int32_t F, const float* row_scale, const float* bias,
                         int32_t relu, void* stream) {
  if (!g) return invalid("graph handle is NULL");
  if (F < 1 || F > (1 << 20)) return invalid("F must be from 1 to 2^20");
  if (g->n == 0) return DG_OK;
  if (!Y || !row_scale || !bias) return invalid("a pointer is NULL");
  return layer_fwd(g, Y, F, row_scale, bias, relu != 0, (cudaStream_t)stream);
}

dg_status_t dg_layer_bwd(dg_graph_t g, const float* dOut, const float* out, int32_t F, const float* row_scale,
                         float* G, float* dbias, void* stream) {
  if (!g) return invalid("graph handle is NULL");
  if (F < 1 || F > (1 << 20)) return invalid("F must be from 1 to 2^20");
  if (!dbias || (g->n > 0 && (!dOut || !row_scale || !G))) return invalid("a pointer is NULL");
  return layer_bwd(g, dOut, out, F, row_scale, G, dbias, (cudaStream_t)stream);
}

// The inputs a and b and the result, with their numbers of elements.
static dg_status_t check_linear(const Graph* g, int32_t N, int32_t K, const float* a, int64_t a_count, const float* b,
                                int64_t b_count, const float* out, int64_t out_count) {
  if (!g) return invalid("graph handle is NULL");
  if (N < 1 || N > (1 << 20) || K < 1 || K > (1 << 20)) return invalid("N and K must be from 1 to 2^20");
  if (g->n > ((int64_t)1 << 31) - 1024) {  // the kernel counts rows, up to a tile beyond the last, in 32 bits
    set_error("the products take at most 2^31 - 1024 rows");
    return DG_ERR_UNSUPPORTED;
  }
  if ((a_count > 0 && !a) || (b_count > 0 && !b) || (out_count > 0 && !out)) return invalid("a pointer is NULL");
  if (overlaps(a, a_count * sizeof(float), out, out_count * sizeof(float)) ||
      overlaps(b, b_count * sizeof(float), out, out_count * sizeof(float)))
    return invalid("the result overlaps an input");
  return DG_OK;
}

dg_status_t dg_linear_fwd(dg_graph_t g, const float* X, int32_t K, const float* W, int32_t N,
                          const float* row_scale, const float* bias, int32_t relu, float* Y, void* stream) {
  const int64_t n = g ? g->n : 0;
  if (dg_status_t st = check_linear(g, N, K, X, n * K, W, (int64_t)N * K, Y, n * N)) return st;
  if (n == 0) return DG_OK;
  return linear_fwd(g, X, K, W, N, row_scale, bias, relu != 0, Y, (cudaStream_t)stream);
}

dg_status_t dg_linear_bwd_input(dg_graph_t g, const float* G, int32_t N, const float* W, int32_t K, float* dX,
                                void* stream) {
  const int64_t n = g ? g->n : 0;
  if (dg_status_t st = check_linear(g, N, K, G, n * N, W, (int64_t)N * K, dX, n * K)) return st;
  if (n == 0) return DG_OK;
  return linear_bwd_input(g, G, N, W, K, dX, (cudaStream_t)stream);
}

dg_status_t dg_linear_bwd_weight(dg_graph_t g, const float* G, int32_t N, const float* X, int32_t K, float* dW,
                                 void* stream) {
  const int64_t n = g ? g->n : 0;
  if (dg_status_t st = check_linear(g, N, K, G, n * N, X, n * K, dW, (int64_t)N * K)) return st;
  if (n == 0) {
    DG_CUDA(cudaMemsetAsync(dW, 0, (size_t)N * K * sizeof(float), (cudaStream_t)stream));
    return DG_OK;
  }
  return linear_bwd_weight(g, G, N, X, K, dW, (cudaStream_t)stream);
}

static dg_status_t check_loss(const Graph* g, int32_t C, int64_t count, const void* stats, bool pointers) {
  if (!g) return invalid("graph handle is NULL");
  if (C < 1 || C > (1 << 20)) return invalid("C must be from 1 to 2^20");
  if (count < 0 || count > ((int64_t)1 << 37)) return invalid("count must be from 0 to 2^37");
  if (count > 0 && g->n == 0) return invalid("the matrix has no rows");
  if (!pointers) return invalid("a pointer is NULL");
  if ((uintptr_t)stats & 7) return invalid("stats must be 8-byte aligned");
  return DG_OK;
}

dg_status_t dg_cross_entropy_fwd(dg_graph_t g, const float* logits, int32_t C, const int64_t* index,
                                 int64_t count, const int64_t* labels, float* stats, float* result,
                                 void* stream) {
  const bool pointers = result && (count <= 0 || (logits && index && labels && stats));
  if (dg_status_t st = check_loss(g, C, count, stats, pointers)) return st;
  return loss_fwd(g, logits, C, index, count, labels, stats, result, (cudaStream_t)stream);
}

dg_status_t dg_cross_entropy_bwd(dg_graph_t g, const float* logits, int32_t C, const int64_t* index,
                                 int64_t count, const int64_t* labels, const float* stats,
                                 const float* result, const float* grad, float* dLogits, void* stream) {
  const bool pointers = (!g || g->n == 0 || dLogits) &&
                        (count <= 0 || (logits && index && labels && stats && result && grad));
  if (dg_status_t st = check_loss(g, C, count, stats, pointers)) return st;
  return loss_bwd(g, logits, C, index, count, labels, stats, result, grad, dLogits, (cudaStream_t)stream);
}

dg_status_t dg_aggregate_bwd(dg_graph_t g, const float* dOut, int32_t F, dg_op_t op, float* dH,
                             void* stream) {
  return run_backward(g, dOut, false, F, op, g && g->self_loops, dH, stream);
}

dg_status_t dg_aggregate_fwd_bf16(dg_graph_t g, const uint16_t* H, int32_t F, dg_op_t op,
                                  float* out, void* stream) {
  return run_forward(g, H, true, F, op, g && g->self_loops, out, stream);
}

dg_status_t dg_aggregate_bwd_bf16(dg_graph_t g, const uint16_t* dOut, int32_t F, dg_op_t op,
                                  float* dH, void* stream) {
  return run_backward(g, dOut, true, F, op, g && g->self_loops, dH, stream);
}

size_t dg_aggregate_host_workspace(dg_graph_t g, int32_t F) {
  if (!g || F < 1) return 0;
  const size_t mat = (((size_t)g->n * (size_t)F * sizeof(float)) + 255) & ~(size_t)255;
  return 4 * (mat > 0 ? mat : 256);
}

// Helper streams (upload, download) and a pool of events per handle, created on first use.
static dg_status_t host_pipeline(Graph* g, size_t events) {
  if (!g->aux_ready) {
    for (int i = 0; i < 2; ++i)
      DG_CUDA(cudaStreamCreateWithFlags(&g->aux_stream[i], cudaStreamNonBlocking));
    g->aux_ready = true;
  }
  if (g->aux_event_count < events) {
    cudaEvent_t* grown = (cudaEvent_t*)realloc(g->aux_events, events * sizeof(cudaEvent_t));
    if (!grown) {
      set_error("out of host memory (event pool)");
      return DG_ERR_INVALID_ARG;
    }
    g->aux_events = grown;
    while (g->aux_event_count < events) {
      DG_CUDA(cudaEventCreateWithFlags(&g->aux_events[g->aux_event_count], cudaEventDisableTiming));
      ++g->aux_event_count;
    }
  }
  return DG_OK;
}

// The feature columns are independent of each other in AP, so the host matrices travel in column
// chunks: chunk c of H is uploaded (a strided copy into a compact n x w matrix) while chunk c-1 is
// being aggregated and the result of chunk c-2 is on its way back; then the same for dOut.  PCIe
// carries both directions at once, so a call costs about max(kernel time, copy time) instead of
// their sum.  Two input and two output chunk buffers alternate.
dg_status_t dg_aggregate_host(dg_graph_t g, const float* H_host, const float* dOut_host,
                              int32_t F, dg_op_t op, float* out_host, float* dH_host,
                              void* device_ws, size_t device_ws_bytes, void* stream) {
  if (!g) return invalid("graph handle is NULL");
  if (F < 1) return invalid("F must be >= 1");
  if (!H_host || !out_host) return invalid("H_host or out_host is NULL");
  if ((dOut_host == nullptr) != (dH_host == nullptr))
    return invalid("dOut_host and dH_host must both be given or both be NULL");
  if (!device_ws || ((uintptr_t)device_ws & 255)) return invalid("device_ws is NULL or misaligned");
  if (device_ws_bytes < dg_aggregate_host_workspace(g, F)) {
    set_error("device_ws smaller than dg_aggregate_host_workspace reports");
    return DG_ERR_WORKSPACE;
  }
  if (dOut_host && !g->transposed) {
    set_error("the backward pass needs dg_graph_transpose first");
    return DG_ERR_NOT_TRANSPOSED;
  }
  if (g->n == 0) return DG_OK;
  // chunk width: 128 columns (one 512-byte row slice) once the matrix is wider than 256 columns
  const int32_t W = F > 256 ? 128 : F;
  const int chunks = (F + W - 1) / W;
  const int tasks = chunks * (dOut_host ? 2 : 1);
  if (dg_status_t st = host_pipeline(g, 1 + 3 * (size_t)tasks)) return st;
  cudaStream_t s = (cudaStream_t)stream;
  cudaStream_t up = g->aux_stream[0], down = g->aux_stream[1];
  cudaEvent_t* ev = g->aux_events;
  cudaEvent_t start = ev[0];
  auto uploaded = [&](int t) { return ev[1 + 3 * t]; };
  auto computed = [&](int t) { return ev[2 + 3 * t]; };
  auto downloaded = [&](int t) { return ev[3 + 3 * t]; };

  const size_t buf = (((size_t)g->n * (size_t)W * sizeof(float)) + 255) & ~(size_t)255;
  char* ws = static_cast<char*>(device_ws);
  float* d_in[2] = {reinterpret_cast<float*>(ws), reinterpret_cast<float*>(ws + buf)};
  float* d_out[2] = {reinterpret_cast<float*>(ws + 2 * buf), reinterpret_cast<float*>(ws + 3 * buf)};
  const size_t host_pitch = (size_t)F * sizeof(float);

  // everything queued on `stream` so far (an earlier call may still use the workspace) comes first
  DG_CUDA(cudaEventRecord(start, s));
  DG_CUDA(cudaStreamWaitEvent(up, start, 0));
  DG_CUDA(cudaStreamWaitEvent(down, start, 0));
  for (int t = 0; t < tasks; ++t) {
    const bool bwd = t >= chunks;
    const int c = bwd ? t - chunks : t;
    const int32_t w = (c + 1) * W <= F ? W : F - c * W;
    const float* src = (bwd ? dOut_host : H_host) + (size_t)c * W;
    float* dst = (bwd ? dH_host : out_host) + (size_t)c * W;
    float* in = d_in[t & 1];
    float* out = d_out[t & 1];
    // upload: the input buffer is free once the kernels of task t-2 have read it
    if (t >= 2) DG_CUDA(cudaStreamWaitEvent(up, computed(t - 2), 0));
    DG_CUDA(cudaMemcpy2DAsync(in, (size_t)w * sizeof(float), src, host_pitch,
                              (size_t)w * sizeof(float), (size_t)g->n, cudaMemcpyHostToDevice, up));
    DG_CUDA(cudaEventRecord(uploaded(t), up));
    // compute: needs the upload, and the output buffer back from the download of task t-2
    DG_CUDA(cudaStreamWaitEvent(s, uploaded(t), 0));
    if (t >= 2) DG_CUDA(cudaStreamWaitEvent(s, downloaded(t - 2), 0));
    if (dg_status_t st = bwd ? dg_aggregate_bwd(g, in, w, op, out, stream)
                             : dg_aggregate_fwd(g, in, w, op, out, stream))
      return st;
    DG_CUDA(cudaEventRecord(computed(t), s));
    // download
    DG_CUDA(cudaStreamWaitEvent(down, computed(t), 0));
    DG_CUDA(cudaMemcpy2DAsync(dst, host_pitch, out, (size_t)w * sizeof(float),
                              (size_t)w * sizeof(float), (size_t)g->n, cudaMemcpyDeviceToHost, down));
    DG_CUDA(cudaEventRecord(downloaded(t), down));
  }
  // `stream` finishing means every copy has finished
  DG_CUDA(cudaStreamWaitEvent(s, downloaded(tasks - 1), 0));
  if (tasks >= 2) DG_CUDA(cudaStreamWaitEvent(s, downloaded(tasks - 2), 0));
  return DG_OK;
}

dg_status_t dg_graph_set_param(dg_graph_t g, const char* name, int64_t value) {
  if (!g || !name) return invalid("graph handle or name is NULL");
  if (!strcmp(name, "heavy_threshold")) {
    if (value < 64 || value > (1 << 30)) return invalid("heavy_threshold must be in [64, 2^30]");
    return replan(g, &g->heavy_threshold, value);
  }
  if (!strcmp(name, "slice_features")) {
    if (value < 0 || value > (1 << 20)) return invalid("slice_features must be in [0, 2^20]");
    g->slice_features = value;
    return DG_OK;
  }
  if (!strcmp(name, "rows_per_block")) {
    if (value < 0 || value > 248) return invalid("rows_per_block must be in [0, 248]");
    if (value == g->rows_per_block) return DG_OK;
    return replan(g, &g->rows_per_block, value);
  }
  if (!strcmp(name, "l2_budget_mb")) {
    if (value < 1 || value > 4096) return invalid("l2_budget_mb must be in [1, 4096]");
    g->l2_budget_bytes = value << 20;
    return DG_OK;
  }
  if (!strcmp(name, "heavy_blocks_per_sm")) {
    if (value < 0 || value > 32) return invalid("heavy_blocks_per_sm must be in [0, 32]");
    g->heavy_blocks_per_sm = value;
    return DG_OK;
  }
  if (!strcmp(name, "self_loops")) {
    if (value != 0 && value != 1) return invalid("self_loops must be 0 or 1");
    g->self_loops = value;
    return DG_OK;
  }
  if (!strcmp(name, "scratch_mb")) {
    if (value < 0 || value > (1 << 20)) return invalid("scratch_mb must be in [0, 2^20]");
    g->scratch_mb = value;
    return DG_OK;
  }
  if (!strcmp(name, "source_blocks")) {
    if (value != 0 && value != 1 && value != 2 && value != 4 && value != 8 && value != 16)
      return invalid("source_blocks must be 0 (automatic), 1, 2, 4, 8 or 16");
    g->source_blocks = value;
    return DG_OK;
  }
  return invalid("unknown parameter name");
}

dg_status_t dg_graph_get_param(dg_graph_t g, const char* name, int64_t* value) {
  if (!g || !name || !value) return invalid("graph handle, name or value is NULL");
  if (!strcmp(name, "heavy_threshold")) {
    *value = g->heavy_threshold > 0 ? g->heavy_threshold : cut_threshold(g);
    return DG_OK;
  }
  if (!strcmp(name, "slice_features")) { *value = g->slice_features; return DG_OK; }
  if (!strcmp(name, "rows_per_block")) { *value = g->rows_per_block; return DG_OK; }
  if (!strcmp(name, "l2_budget_mb")) { *value = g->l2_budget_bytes >> 20; return DG_OK; }
  if (!strcmp(name, "source_blocks")) { *value = g->source_blocks; return DG_OK; }
  if (!strcmp(name, "self_loops")) { *value = g->self_loops; return DG_OK; }
  if (!strcmp(name, "scratch_mb")) { *value = g->scratch_mb; return DG_OK; }
  if (!strcmp(name, "heavy_blocks_per_sm")) { *value = g->heavy_blocks_per_sm; return DG_OK; }
  if (!strcmp(name, "expired_waits")) return linear_expired(value);
  return invalid("unknown parameter name");
}

int64_t dg_kernel_launch_count(void) { return g_launches.load(std::memory_order_relaxed); }

const char* dg_last_error(void) { return g_last_error; }

const char* dg_version(void) { return "libdgagg 0.8 sm_100a"; }

}  // extern "C"
