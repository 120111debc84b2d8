// Graph ingest kernels: how rows are shared out among warps, split pointers, CSR validation.
// All integer work; nothing here waits on another block.
#include "dg_internal.cuh"

namespace dg {
namespace {

constexpr int kBlock = 256;

// Boundary c of a plan lies at cost c * chunk_cost, where reaching entry k of row r has cost
// k + row_cost * r: a row costs its entries and row_cost for its pointer, its index batch and its store,
// so that runs of short or empty rows are shared out too, and no chunk has more than 31 rows.  A boundary
// inside a row of up to `threshold` entries, and the last of the boundaries inside a longer row, move to
// the end of the row; the others stay inside the row, spread evenly over what follows the first of
// them, at multiples of 32 entries.  So a chunk that begins inside a row is a piece of that row alone.
// (A malformed row pointer gives meaningless chunks here, and no access outside the arrays.)
__global__ void plan_kernel(const int64_t* __restrict__ ptr, int64_t n, int64_t nnz, int64_t chunk_cost,
                            int64_t row_cost, int64_t threshold, int64_t count, Chunk* __restrict__ chunks,
                            CutRow* __restrict__ cuts, int64_t max_cuts, int32_t* __restrict__ totals) {
  const int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (c > count) return;
  Chunk out{(int32_t)n, (int32_t)nnz, -1, 0};
  const int64_t d = c * chunk_cost;
  if (c < count) {
    int64_t lo = 0, hi = n;  // the last row r with ptr[r] + row_cost * r <= d
    while (hi - lo > 1) {
      const int64_t mid = (lo + hi) >> 1;
      if (__ldg(ptr + mid) + row_cost * mid <= d) lo = mid; else hi = mid;
    }
    const int64_t start = __ldg(ptr + lo), len = __ldg(ptr + lo + 1) - start;
    const int64_t base = start + row_cost * lo;
    if (d <= base) {
      out.row = (int32_t)lo;
      out.pos = (int32_t)start;
    } else {
      out.row = (int32_t)(lo + 1);
      out.pos = (int32_t)(start + len);
      const int64_t first = base / chunk_cost + 1, last = (base + len) / chunk_cost;
      if (len > threshold && c < last) {
        const int64_t off = first * chunk_cost - base, j = c - first, m = last - first;
        const int64_t cut = (off + j * ((len - off) / m) + 31) & ~(int64_t)31;
        out.row = (int32_t)lo;
        out.pos = (int32_t)(start + cut);  // cut < len: the pieces are at least chunk_cost >= 32 long
        out.slot = atomicAdd(totals + 0, 1);
        if (j == 0) {
          const int32_t i = atomicAdd(totals + 1, 1);
          atomicMax(totals + 2, (int32_t)m);
          if (i < max_cuts) cuts[i] = CutRow{(int32_t)lo, (int32_t)c, (int32_t)m, 0};
        }
      }
    }
  }
  chunks[c] = out;
}

// flags: bit 0 rowptr[0] != 0, bit 1 rowptr decreasing, bit 2 rowptr[n] != nnz,
//        bit 3 colidx out of range
__global__ void check_csr_kernel(const int64_t* __restrict__ rowptr, const int32_t* __restrict__ colidx,
                                 int64_t n, int64_t nnz, int32_t* __restrict__ flags) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  const int64_t first = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  int f = 0;
  for (int64_t v = first; v < n; v += stride)
    if (rowptr[v + 1] < rowptr[v]) f |= 2;
  if (first == 0) {
    if (rowptr[0] != 0) f |= 1;
    if (rowptr[n] != nnz) f |= 4;
  }
  // 16-byte loads of the caller's array, which is only 4-byte aligned in general
  const int64_t head = nnz < 4 ? nnz : (int64_t)((16 - ((uintptr_t)colidx & 15)) & 15) / 4;
  const int64_t quads = (nnz - head) / 4;
  const uint32_t top = (uint32_t)n;
  const int4* body = reinterpret_cast<const int4*>(colidx + head);
#pragma unroll 4
  for (int64_t k = first; k < quads; k += stride) {
    const int4 u = __ldcs(body + k);
    if ((uint32_t)u.x >= top || (uint32_t)u.y >= top || (uint32_t)u.z >= top || (uint32_t)u.w >= top) f |= 8;
  }
  if (first < head && (uint32_t)colidx[first] >= top) f |= 8;
  const int64_t tail = head + 4 * quads + first;
  if (tail < nnz && (uint32_t)colidx[tail] >= top) f |= 8;
  if (f) atomicOr(flags, f);
}

// split[b * n + v] for b = 0..kFineBlocks: the first position of segment v whose id is
// >= b * fine_rows, by binary search (the segment must be sorted ascending).
__global__ void split_kernel(const int64_t* __restrict__ ptr, const int32_t* __restrict__ idx,
                             int64_t n, int64_t fine_rows, int32_t* __restrict__ split,
                             const int32_t* __restrict__ malformed) {
  if (malformed && *malformed) return;
  const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= (int64_t)(kFineBlocks + 1) * n) return;
  const int64_t b = t / n, v = t - b * n;
  int64_t lo = ptr[v], hi = ptr[v + 1];
  if (b == 0) { split[t] = (int32_t)lo; return; }
  if (b == kFineBlocks) { split[t] = (int32_t)hi; return; }
  const int64_t bound = b * fine_rows;
  while (lo < hi) {
    const int64_t mid = (lo + hi) >> 1;
    if ((int64_t)__ldg(idx + mid) < bound) lo = mid + 1; else hi = mid;
  }
  split[t] = (int32_t)lo;
}

// One warp per segment: sets *flag when two adjacent ids of a segment are out of order.
__global__ void sorted_check_kernel(const int64_t* __restrict__ ptr,
                                    const int32_t* __restrict__ idx, int64_t n,
                                    int32_t* __restrict__ flag,
                                    const int32_t* __restrict__ malformed) {
  if (malformed && *malformed) return;  // row pointers that may lie outside idx
  const int64_t v = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  if (v >= n) return;
  const int lane = threadIdx.x & 31;
  const int64_t lo = ptr[v], hi = ptr[v + 1];
  int bad = 0;
  for (int64_t k = lo + 1 + lane; k < hi; k += 32)
    if (__ldg(idx + k - 1) > __ldg(idx + k)) bad = 1;
  if (bad) atomicOr(flag, 1);
}

inline unsigned blocks_for(int64_t items) { return (unsigned)((items + kBlock - 1) / kBlock); }

}  // namespace

bool wants_split(int64_t n, int64_t nnz) {
  return n >= 4096 && nnz >= kBlockingMinAvgLen * n &&
         (int64_t)(kFineBlocks + 1) * n < ((int64_t)1 << 40);
}

// Fills the split pointers of one direction and raises *unsorted_flag (device) when a segment
// is not sorted ascending, in which case the pointers must not be used.  `malformed` (device, may be
// nullptr): non-zero when the CSR failed its check, which was queued before this.
dg_status_t build_split(const int64_t* ptr, const int32_t* idx, int64_t n, int64_t fine_rows,
                        int32_t* split, int32_t* unsorted_flag, const int32_t* malformed, cudaStream_t s) {
  DG_CUDA(cudaMemsetAsync(unsorted_flag, 0, sizeof(int32_t), s));
  sorted_check_kernel<<<blocks_for(n * 32), kBlock, 0, s>>>(ptr, idx, n, unsorted_flag, malformed);
  DG_CUDA(cudaGetLastError());
  split_kernel<<<blocks_for((int64_t)(kFineBlocks + 1) * n), kBlock, 0, s>>>(ptr, idx, n, fine_rows,
                                                                            split, malformed);
  DG_CUDA(cudaGetLastError());
  count_launches(2);
  return DG_OK;
}

// The chunks of one direction (the arrays of `plan` are sized by its count); asynchronous.
dg_status_t build_plan(const int64_t* ptr, int64_t n, int64_t nnz, int64_t chunk_cost, int64_t row_cost,
                       int64_t threshold, const Plan& plan, cudaStream_t s) {
  DG_CUDA(cudaMemsetAsync(plan.totals, 0, kTotalsPerPlan * sizeof(int32_t), s));
  plan_kernel<<<blocks_for(plan.count + 1), kBlock, 0, s>>>(ptr, n, nnz, chunk_cost, row_cost, threshold, plan.count,
                                                            plan.chunks, plan.cuts, plan.max_cuts,
                                                            plan.totals);
  DG_CUDA(cudaGetLastError());
  count_launches(1);
  return DG_OK;
}

// Queues the check of the borrowed CSR; *flags (device) collects what is wrong with it.
dg_status_t check_csr(const Graph* g, int32_t* flags, cudaStream_t s) {
  DG_CUDA(cudaMemsetAsync(flags, 0, sizeof(int32_t), s));
  const int64_t items = g->nnz / 4 > g->n ? g->nnz / 4 : g->n;
  int64_t blocks = (items + kBlock - 1) / kBlock;
  if (blocks > (int64_t)g->sm_count * 16) blocks = (int64_t)g->sm_count * 16;
  if (blocks < 1) blocks = 1;
  check_csr_kernel<<<(unsigned)blocks, kBlock, 0, s>>>(g->rowptr, g->colidx, g->n, g->nnz, flags);
  DG_CUDA(cudaGetLastError());
  count_launches(1);
  return DG_OK;
}

}  // namespace dg
