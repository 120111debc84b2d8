// Internal declarations shared by the translation units of libdgagg (not part of the ABI).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>

#include "dg.h"

namespace dg {

// One warp's share of a pass over the CSR rows (or CSC columns): the entries [pos, next chunk's
// pos), which belong to the rows from `row` up to the next chunk's row.  Chunks hold about the same
// number of entries.  They begin at row starts, except inside rows longer than the split threshold:
// such a row is cut, and a chunk that begins inside a row (slot >= 0) leaves its part of that row in
// slot `slot` of a scratch array instead of in the output; a second small launch adds the slots of
// every cut row to what its first chunk stored, in order (see dg_aggregate.cu).
struct Chunk {
  int32_t row, pos, slot, pad;
};
// A cut row: the chunks first .. first + count - 1 begin inside it.
struct CutRow {
  int32_t row, first, count, pad;
};
// The chunks of one direction; the arrays are owned by the handle.
struct Plan {
  Chunk* chunks = nullptr;    // count + 1 entries, the last one is (n, nnz)
  CutRow* cuts = nullptr;     // the cut rows, in any order
  int32_t* totals = nullptr;  // device: [0] slots, [1] cut rows, [2] most slots of a row
  int64_t count = 0;
  int64_t max_slots = 0, max_cuts = 0;  // bounds known from n and nnz alone
  int32_t slots = -1, cut_rows = -1, most_pieces = -1;  // the totals, or -1 while they are on their way to the host
};

// Device counters of a handle, and their order in the pinned copy.  There are two sets of plan totals, rows' then
// columns', used in turn: until new plans are finished the old ones stay whole.
enum { kFlags, kUnsorted, kTotals, kTotalsPerPlan = 3, kCounters = kTotals + 4 * kTotalsPerPlan };
struct HostCounters {
  int32_t v[kCounters];
};

}  // namespace dg

// What a handle records.  CSR and CSC arrays are borrowed; the small arrays below are owned.
struct dg_graph {
  int64_t n = 0, nnz = 0;
  const int64_t* rowptr = nullptr;
  const int32_t* colidx = nullptr;
  const float* edge_w = nullptr;

  // one block of device memory behind the arrays below, and one behind the two plans
  void* owned = nullptr;
  size_t owned_bytes = 0;
  void* plan_memory = nullptr;
  size_t plan_bytes = 0;
  dg::Plan row_plan, col_plan;   // CSR rows (forward), CSC columns (backward)
  int32_t totals_set = 0;        // which totals in `counters` are theirs

  int32_t* counters = nullptr;   // kCounters device words, see the enum below

  // Source blocking: the neighbour ids are cut into kFineBlocks ranges of fine_rows ids;
  // split[b * n + v] is the first position of segment v whose neighbour id is >= b * fine_rows
  // (entry kFineBlocks is the segment end).  Built only for graphs whose rows are long and
  // sorted; nullptr otherwise.  split_csr is owned, split_csc lives in the caller's CSC storage.
  int32_t* split_csr = nullptr;
  int32_t* split_csc = nullptr;
  int64_t fine_rows = 0;

  // dg_aggregate_host: helper streams (upload, download) and events, created on first use
  bool aux_ready = false;
  cudaStream_t aux_stream[2] = {nullptr, nullptr};
  cudaEvent_t* aux_events = nullptr;  // malloc'ed pool, aux_event_count entries
  size_t aux_event_count = 0;

  // pinned copy of `counters`; col_plan's totals arrive in it some time after a transposition
  dg::HostCounters* host = nullptr;
  cudaEvent_t col_totals_ready = nullptr;  // recorded behind that copy

  bool transposed = false;
  const int64_t* colptr = nullptr;
  const int32_t* rowidx_T = nullptr;
  const float* w_T = nullptr;
  const int32_t* perm = nullptr;
  const float* mean_scale_T = nullptr;  // w_T[q] / (deg(rowidx_T[q]) + self_loops): edge factor of the mean's backward
  int64_t self_loops = 0;        // 1: every vertex is its own in-neighbour with weight 1
  int64_t self_loops_in_csc = 0; // value mean_scale_T was built with

  // set on a handle made by dg_graph_reorder: arrays inside the caller's reorder storage
  const int32_t* new_of_old = nullptr;   // n: new id of every old vertex
  const int32_t* reorder_pos = nullptr;  // nnz: old CSR position of every new position

  int device = 0;
  int sm_count = 148;
  size_t l2_bytes = 0;
  int64_t heavy_threshold = 0;   // rows longer than this are cut; 0 = automatic
  int64_t slice_features = 0;    // 0 = automatic
  int64_t rows_per_block = 0;    // 0 = from the average row length
  int64_t heavy_blocks_per_sm = 0;  // recorded for dg_graph_get_param, no effect
  int64_t l2_budget_bytes = 0;   // bytes of the gathered matrix one launch may keep L2-resident
  int64_t source_blocks = 0;     // 0 = automatic, else 1, 2, 4, 8 or 16
  int64_t scratch_mb = 4096;     // most MiB of a scratch block of a call; 0: calls take no memory
};

namespace dg {

using Graph = ::dg_graph;

// A position in the edge arrays while a kernel steps through them in batches: all are below 2^31, and a step past
// the last one overflows a signed 32-bit number.
using Position = uint32_t;

constexpr int kFineBlocks = 16;          // finest cut of the neighbour ids for source blocking
constexpr int64_t kBlockingMinAvgLen = 64;  // split pointers are built when nnz >= 64 n

// One direction of AP as the kernels see it: out[r] = rs_r * sum_k s_k * X[idx[k]],
// s_k = w[k] (1 when w is absent).
struct ApArgs {
  const int64_t* ptr;         // n+1 segment pointers (rowptr or colptr)
  const int32_t* idx;         // neighbour ids (colidx or rowidx_T)
  const float* w;             // per-edge weight or nullptr
  const void* X;              // n x F input: fp32, or bf16 when x_bf16 is set
  uint32_t row_bytes;         // distance between its rows
  int32_t x_bf16;
  float* Y;                   // n x F output
  int32_t narrow_store;       // 1: the rows of Y cannot take the vector width that X is read with
  const Chunk* chunks;        // chunk_count + 1
  int32_t chunk_count;
  float* partial;             // slots x F: the parts of cut rows; nullptr: left out, see dg_pieces.cu
  int64_t n;
  int32_t F;
  int32_t slice_f;            // features per slice (multiple of the vector width)
  int32_t mean_rows;          // 1: multiply the finished row by 1/(segment length)
  const int32_t* seg_lo;      // source-blocked pass: first and one-past-last position of every
  const int32_t* seg_hi;      //   segment's piece (n entries each); nullptr = whole segments
  int32_t accumulate;         // source-blocked pass after the first: add to what Y holds
  int32_t overlap;            // host side: launch while the previous kernel (the copy) drains, see launch_kernel
  int32_t few_blocks;         // host side: the grid is small, see ap_kernel
  int32_t long_rows;          // host side: the mean degree is 24 or more
  int32_t mean_factors;       // host side: w are the factors 1 / deg (+ 1) of the mean's backward pass alone
};

// Implicit self loops (every vertex its own neighbour with weight 1): row r also receives
// ss_r * X[r], once (not in accumulating passes).  self_ptr is the CSR row pointer, in both
// directions (the in-degree belongs to the vertex, not to the segment the kernel walks);
// nullptr = no self loops.  self_mean: ss_r = 1 / (in-degree(r) + 1) instead of 1, and
// mean_rows scales by the same factor instead of 1 / (segment length).  A parameter of its own,
// passed only to the kernels compiled for self loops.
struct SelfArgs {
  const int64_t* self_ptr;
  int32_t self_mean;
};

// One launch of the aggregation kernels in the shape aggregate_run chose (dg_aggregate.cu,
// dg_aggregate_self.cu).
dg_status_t launch_plain(const ApArgs& a, int vec, int slices, cudaStream_t s);
dg_status_t launch_with_self_loops(const ApArgs& a, const SelfArgs& sa, int vec, int slices,
                                   cudaStream_t s);
// Records the calling thread's last error message (printf-style, truncated to a fixed buffer:
// nothing on an error path allocates, so nothing can throw across the C boundary).
void set_error(const char* fmt, ...) __attribute__((format(printf, 1, 2)));
dg_status_t cuda_fail(cudaError_t e, const char* what);
void count_launches(int64_t k);

// Launches `kernel`; with `overlap` its blocks may start while the kernel before it on the stream drains (and
// after all of that one's blocks have started), so it must begin with cudaGridDependencySynchronize(), which
// waits for that kernel's end and for its writes.  For kernels of a few microseconds the gap between two
// launches is worth closing (forward + backward with copies and joins, 1.2 M edges, F = 47: 85 -> 75 us; with a
// join, 65 k edges, F = 64: 20.5 -> 18.8 us).
template <typename... P, typename... A>
cudaError_t launch_kernel(void (*kernel)(P...), dim3 grid, int block, size_t smem, cudaStream_t s, bool overlap,
                          const A&... args) {
  cudaLaunchAttribute attribute{};
  attribute.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attribute.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t config{};
  config.gridDim = grid;
  config.blockDim = dim3((unsigned)block);
  config.dynamicSmemBytes = smem;
  config.stream = s;
  config.attrs = &attribute;
  config.numAttrs = overlap ? 1 : 0;
  return cudaLaunchKernelEx(&config, kernel, args...);
}
template <typename... P, typename... A>
cudaError_t launch_kernel(void (*kernel)(P...), dim3 grid, int block, cudaStream_t s, bool overlap, const A&... args) {
  return launch_kernel(kernel, grid, block, (size_t)0, s, overlap, args...);
}

#define DG_CUDA(call)                                          \
  do {                                                         \
    cudaError_t e__ = (call);                                  \
    if (e__ != cudaSuccess) return dg::cuda_fail(e__, #call);  \
  } while (0)

// Makes `device` current for a scope: handles are destroyed and their knobs set with any device current (a garbage
// collector decides when), and waiting and stream-ordered calls act on the current one.
class DeviceScope {
 public:
  explicit DeviceScope(int device) {
    if (cudaGetDevice(&before_) != cudaSuccess) before_ = device;
    if (before_ != device) cudaSetDevice(device);
    device_ = device;
  }
  ~DeviceScope() {
    if (before_ != device_) cudaSetDevice(before_);
  }
  DeviceScope(const DeviceScope&) = delete;
  DeviceScope& operator=(const DeviceScope&) = delete;

 private:
  int before_ = 0, device_ = 0;
};

// dg_pool.cu: device memory of the library itself
cudaError_t pool_open(int device);   // one per handle
void pool_close(int device);
cudaError_t pool_wait(int device);   // waits for the device, then frees what was retired before
cudaError_t pool_alloc(int device, size_t bytes, cudaStream_t s, void** out);
void pool_free(void* p, cudaStream_t s);
// Scratch of a call, within the handle's limit; a call has to do without it when there is none.
cudaError_t scratch_alloc(const Graph* g, size_t bytes, cudaStream_t s, void** out);
void pool_retire(int device, void* p, size_t bytes);  // kernels on any stream may still use it
cudaError_t pinned_counters(HostCounters** out);
void pinned_counters_retire(int device, HostCounters* p);

// dg_graph.cu
dg_status_t build_plan(const int64_t* ptr, int64_t n, int64_t nnz, int64_t chunk_cost, int64_t row_cost,
                       int64_t threshold, const Plan& plan, cudaStream_t s);
dg_status_t check_csr(const Graph* g, int32_t* flags, cudaStream_t s);
bool wants_split(int64_t n, int64_t nnz);
dg_status_t build_split(const int64_t* ptr, const int32_t* idx, int64_t n, int64_t fine_rows,
                        int32_t* split, int32_t* unsorted_flag, const int32_t* malformed, cudaStream_t s);

// dg_layer.cu
dg_status_t layer_fwd(const Graph* g, float* Y, int32_t F, const float* scale, const float* bias, bool relu,
                      cudaStream_t s);
dg_status_t layer_bwd(const Graph* g, const float* dOut, const float* out, int32_t F, const float* scale,
                      float* G, float* dbias, cudaStream_t s);

// dg_linear.cu
dg_status_t linear_fwd(const Graph* g, const float* X, int32_t K, const float* W, int32_t N, const float* scale,
                       const float* bias, bool relu, float* Y, cudaStream_t s);
dg_status_t linear_bwd_input(const Graph* g, const float* G, int32_t N, const float* W, int32_t K, float* dX,
                             cudaStream_t s);
dg_status_t linear_bwd_weight(const Graph* g, const float* G, int32_t N, const float* X, int32_t K, float* dW,
                              cudaStream_t s);
dg_status_t linear_expired(int64_t* blocks);  // blocks that gave up a wait, on the current device

// dg_loss.cu
dg_status_t loss_fwd(const Graph* g, const float* logits, int32_t C, const int64_t* index, int64_t count,
                     const int64_t* labels, float* stats, float* result, cudaStream_t s);
dg_status_t loss_bwd(const Graph* g, const float* logits, int32_t C, const int64_t* index, int64_t count,
                     const int64_t* labels, const float* stats, const float* result, const float* grad,
                     float* d, cudaStream_t s);

// dg_transpose.cu
void transpose_sizes(int64_t n, int64_t nnz, bool weighted, size_t* csc_bytes,
                     size_t* scratch_bytes);
dg_status_t transpose_run(Graph* g, void* csc, void* scratch, cudaStream_t s);
dg_status_t refresh_csc_weights(Graph* g, cudaStream_t s);
// dg_api.cu: what follows every transposition (the columns' plan, its totals on their way to the host)
dg_status_t finish_transpose(Graph* g, cudaStream_t s);
// the stable radix sort behind it, for other pre-processing steps (see dg_transpose.cu)
struct SortPlan { int digit_bits; int passes; };
SortPlan sort_plan(int64_t key_range);
void sort_scratch_sizes(int64_t count, size_t* hist_bytes, size_t* sums_bytes);
dg_status_t sort_pairs(const uint32_t* keys_in, const uint32_t* vals_in, int64_t count, SortPlan plan,
                       uint32_t* const keys_buf[2], uint32_t* vals_final, uint32_t* vals_tmp,
                       uint32_t* hist, uint32_t* sums, const uint32_t** sorted_keys,
                       cudaStream_t s);
dg_status_t pointers_from_sorted_keys(const uint32_t* sorted, int64_t count, int64_t n,
                                      int64_t* ptr, cudaStream_t s);
dg_status_t expand_rows(const int64_t* rowptr, int64_t n, int64_t nnz, const int32_t* map,
                        uint32_t* out, cudaStream_t s);

// Whether a call first copies a gathered matrix into padded rows, and the copy (dg_aggregate.cu).
bool worth_padding(const Graph* g, int32_t F, int elem_bytes, int vec);
dg_status_t pad_rows(const Graph* g, const void* X, int32_t F, int elem_bytes, const int64_t* mean_ptr, int mean_self,
                     cudaStream_t s, void** copy, int64_t* ld);
// Scratch for the parts of cut rows, and their join.  nullptr when the plan cuts none, or when there is no memory
// (`missing`): then the pieces are left out of the main kernels and added by add_pieces (dg_pieces.cu).
float* take_partial(const Graph* g, const Plan& plan, int64_t floats_per_slot, cudaStream_t s, bool* missing);
struct PieceArgs {
  const Chunk* chunks;     // the first four come from the plan
  const CutRow* cuts;
  const int32_t* totals;
  int32_t max_cuts;
  int32_t F;
  const int32_t* idx;      // nullptr: nothing is gathered (copyrhs)
  const int32_t* perm;     // over the CSC: CSR position of every entry
  const void* X;           // gathered rows, ldx elements apart
  int64_t ldx;
  const float* w;          // factor of the entry (sum and mean calls), in the order walked
  const float* Y;          // edge operand, edge_cols = 1 or F columns, in CSR order
  const int32_t* arg;      // gradient of max / min
  const int64_t* mean_ptr; // rows divided by their length here + mean_self
  float* out;
  int32_t* arg_out;
  int32_t bf16, edge_cols, bin, red, gradient, mean_self;
};
dg_status_t add_pieces(const Graph* g, const Plan& plan, PieceArgs a, cudaStream_t s);
dg_status_t join_cut_rows(const Graph* g, const Plan& plan, const float* partial, int32_t F, float* Y,
                          cudaStream_t s);
// dg_edge_grad.cu
dg_status_t edge_grad_run(const Graph* g, const float* H, const float* dOut, int32_t F, int row_scale,
                          float* dW, cudaStream_t s);
// dg_api.cu: the plan of the CSC, with its totals if they have arrived
const Plan& column_plan(Graph* g);

// dg_aggregate.cu
dg_status_t aggregate_run(const Graph* g, const ApArgs& a, const SelfArgs& sa, const Plan& plan,
                          const int32_t* split, cudaStream_t s);
// sum_k w_k X[idx[k]] over the CSR rows or the CSC columns with those kernels (dg_api.cu); w in
// the order of that direction or nullptr, no self loops.
dg_status_t aggregate_sum(Graph* g, bool over_csc, const float* w, const float* X, int32_t F,
                          float* Y, cudaStream_t s);

}  // namespace dg
