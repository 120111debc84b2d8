// What the kernels of the general aggregation primitive share (dg_general_fwd.cu, dg_general_bwd.cu,
// dg_edge_grad.cu): arguments, the message and its derivatives, the walk over a chunk.
//
// Work decomposition as in dg_aggregate_kernels.cuh: a warp takes one chunk of the plan, G lanes spread
// along the features take one edge, the 32 / G lane groups take different edges, and several steps of
// loads are in flight before the first use.  A grid row covers G * VEC features (at most 128).
// With a warp per row instead, and a block per row of over 1024 edges, the longest rows set the time of
// skewed graphs, and without warp-uniform indices the kernels were short of registers: copylhs / max on
// 31 M edges, F = 100: 2.41 -> 1.62 ms.
//
// Determinism: every output element is produced by one warp in a fixed order (the pieces of a cut row are
// merged in order by a second launch); the extremum of max / min is chosen on (message, edge position)
// pairs, equal messages going to the lowest position.  No floating-point atomics.
#ifndef DG_GENERAL_CUH_
#define DG_GENERAL_CUH_
#include "dg_internal.cuh"

namespace dg {

constexpr int kGenBlock = 256;
constexpr int kGenWarps = kGenBlock / 32;

enum { kCopyLhs = DG_BIN_COPY_LHS, kCopyRhs = DG_BIN_COPY_RHS, kAdd = DG_BIN_ADD,
       kSub = DG_BIN_SUB, kMul = DG_BIN_MUL, kDiv = DG_BIN_DIV };
enum { kSum = DG_RED_SUM, kMax = DG_RED_MAX, kMin = DG_RED_MIN };
// the edge operand: absent, one scalar per edge, F values per edge
enum { kNoEdge = 0, kEdgeScalar = 1, kEdgeFull = 2 };

struct GenArgs {
  const Chunk* chunks;
  int32_t chunk_count;
  const int64_t* ptr;     // n+1 segment pointers: rowptr, or colptr in the pass over the CSC
  const int32_t* idx;     // colidx, or rowidx_T
  const int32_t* perm;    // CSC pass: CSR position of every CSC entry
  const float* X;         // rows that are gathered or, in the edge gradient, read once per row: fV, dO
  int64_t ldx;            // floats between rows of X
  const float* V;         // edge gradient: fV, gathered
  const float* Y;         // edge features in CSR position order
  const int32_t* arg;     // n x F edge positions of the extrema (max / min)
  uint32_t* mask;         // per edge `words` words: bit j of word w is feature f_lo + 32 w + j, see dg_general_bwd.cu
  int32_t words;
  int32_t f_lo;           // first feature of the mask
  float* out;             // n x F, or nnz x cols in the edge gradient
  int32_t* arg_out;
  float* partial;         // slots x F: the parts of cut rows
  int32_t skip_pieces;    // no memory for them: left out, see dg_pieces.cu
  int32_t* partial_arg;   // and their edge positions (max / min)
  int32_t F, cols;
  int32_t log_g;          // lanes per edge = 1 << log_g
  int32_t vec;            // host side: floats per load
  int32_t first_slice;    // slice of the launch's first grid row
  int32_t slices;         // host side: grid rows; 0 = all slices
  // one launch of a source-blocked call: the piece [seg_lo[v], seg_hi[v]) of every row (nullptr: whole
  // rows), and whether out (and arg_out) already hold the result of the earlier pieces
  const int32_t* seg_lo;
  const int32_t* seg_hi;
  int32_t accumulate;
};

// dg_general_fwd.cu, dg_general_bwd.cu: one launch of the kernel for an operator pair
dg_status_t launch_general_fwd(const GenArgs& a, int bin, int red, cudaStream_t s);
dg_status_t launch_general_dv(const GenArgs& a, int bin, int red, cudaStream_t s);
dg_status_t launch_general_de(const GenArgs& a, int bin, int red, cudaStream_t s);
dg_status_t launch_arg_mask(const GenArgs& over_rows, cudaStream_t s);
dg_status_t join_extrema(const Graph* g, const Plan& plan, const GenArgs& a, int red, cudaStream_t s);

#ifdef __CUDACC__
namespace {

constexpr unsigned kAll = 0xffffffffu;
struct True { static constexpr bool value = true; };
struct False { static constexpr bool value = false; };

// one fp32 IEEE operation, never contracted into a neighbouring add
template <int BIN>
__device__ __forceinline__ float message(float x, float y) {
  if (BIN == kCopyLhs) return x;
  if (BIN == kCopyRhs) return y;
  if (BIN == kAdd) return __fadd_rn(x, y);
  if (BIN == kSub) return __fsub_rn(x, y);
  if (BIN == kMul) return __fmul_rn(x, y);
  return __fdiv_rn(x, y);
}
template <int BIN>
__device__ __forceinline__ float d_dx(float y) {
  if (BIN == kCopyRhs) return 0.f;
  if (BIN == kMul) return y;
  if (BIN == kDiv) return __fdiv_rn(1.f, y);
  return 1.f;
}
template <int BIN>
__device__ __forceinline__ float d_dy(float x, float y) {
  if (BIN == kCopyLhs) return 0.f;
  if (BIN == kSub) return -1.f;
  if (BIN == kMul) return x;
  if (BIN == kDiv) return -__fdiv_rn(x, __fmul_rn(y, y));
  return 1.f;
}

// (value, position) of the better of two candidates; position < 0 means "none"
template <int RED>
__device__ __forceinline__ void take_better(float& best, int32_t& best_k, float m, int32_t k) {
  if (k < 0) return;
  const bool better = RED == kMax ? m > best : m < best;
  if (best_k < 0 || better || (m == best && k < best_k)) {
    best = m;
    best_k = k;
  }
}

// loads VEC consecutive floats (ints) into dst[0..VEC): cached, or streaming (read once)
template <int VEC>
__device__ __forceinline__ void load_vec(float* dst, const float* src) {
  if constexpr (VEC == 4) {
    const float4 v = __ldg(reinterpret_cast<const float4*>(src));
    dst[0] = v.x; dst[1] = v.y; dst[2] = v.z; dst[3] = v.w;
  } else if constexpr (VEC == 2) {
    const float2 v = __ldg(reinterpret_cast<const float2*>(src));
    dst[0] = v.x; dst[1] = v.y;
  } else {
    dst[0] = __ldg(src);
  }
}
template <int VEC>
__device__ __forceinline__ void load_vec(int32_t* dst, const int32_t* src) {
  load_vec<VEC>(reinterpret_cast<float*>(dst), reinterpret_cast<const float*>(src));
}
template <int VEC>
__device__ __forceinline__ void stream_vec(float* dst, const float* src) {
  if constexpr (VEC == 4) {
    const float4 v = __ldcs(reinterpret_cast<const float4*>(src));
    dst[0] = v.x; dst[1] = v.y; dst[2] = v.z; dst[3] = v.w;
  } else if constexpr (VEC == 2) {
    const float2 v = __ldcs(reinterpret_cast<const float2*>(src));
    dst[0] = v.x; dst[1] = v.y;
  } else {
    dst[0] = __ldcs(src);
  }
}
// *p if `wanted`, else `other`.  A predicated load: written as an if, the loads of a step become branches
// that are taken, and waited for, one after the other.
__device__ __forceinline__ float load_if(bool wanted, const float* p, float other) {
  asm("{\n\t.reg .pred w;\n\tsetp.ne.u32 w, %2, 0;\n\t@w ld.global.nc.f32 %0, [%1];\n\t}"
      : "+f"(other)
      : "l"(p), "r"((uint32_t)wanted));
  return other;
}

// Walks the warp's chunk row by row and each row in batches of up to 32 edges:
//   first(u, k); { begin(r); batch(u, k, b, cnt, next_u, next_k) ...; end(r, slot) } ...
// u (k): lane i holds the neighbour id (CSR position, with PERM) of edge b + i, 0 in lanes without an edge;
// next_u, next_k: those of the batch that follows, also across rows (meaningless but valid ids after the
// last one), for loads that start a batch ahead; first() gets the ids of the first batch.  slot >= 0: the
// row's part belongs to that slot.  Everything but the ids is the same in all lanes, and the shuffle of the warp's
// number lets the compiler know (uniform registers; see dg_aggregate_kernels.cuh).
template <bool IDX, bool PERM, class First, class Begin, class Batch, class End>
__device__ __forceinline__ void walk_chunk(const GenArgs& a, First first, Begin begin, Batch batch, End end) {
  const int lane = threadIdx.x & 31;
  const int chunk = blockIdx.x * kGenWarps + __shfl_sync(kAll, (int)(threadIdx.x >> 5), 0);
  if (chunk >= a.chunk_count) return;
  const int4 here = __ldg(reinterpret_cast<const int4*>(a.chunks) + chunk);
  if (here.z >= 0 && a.skip_pieces) return;
  const int4 next = __ldg(reinterpret_cast<const int4*>(a.chunks) + chunk + 1);
  const int nrows = here.z >= 0 ? 1 : next.x - here.x + (next.z >= 0 ? 1 : 0);
  int my_lo = 0, my_hi = 0;
  if (lane < nrows) {
    const int64_t r = here.x + lane;
    my_lo = max(a.seg_lo ? __ldg(a.seg_lo + r) : (int)__ldg(a.ptr + r), here.y);
    my_hi = min(a.seg_hi ? __ldg(a.seg_hi + r) : (int)__ldg(a.ptr + r + 1), next.y);
  }
  const unsigned work = __ballot_sync(kAll, my_hi > my_lo);
  int qi = work ? __ffs(work) - 1 : 32;
  Position qb = 0, qhi = 0;  // the batch that is fetched next
  int32_t cur_u = 0, nxt_u = 0, cur_k = 0, nxt_k = 0;
  auto fetch = [&](int32_t& u, int32_t& k) {
    const bool mine = qb + lane < qhi;
    if (IDX) u = mine ? __ldcs(a.idx + qb + lane) : 0;
    if (PERM) k = mine ? __ldcs(a.perm + qb + lane) : 0;
  };
  auto step_q = [&]() {
    qb += 32;
    if (qb >= qhi) {
      const unsigned rest = qi >= 31 ? 0u : (work & ~((2u << qi) - 1u));
      qi = rest ? __ffs(rest) - 1 : 32;
      if (qi < 32) {
        qb = __shfl_sync(kAll, my_lo, qi);
        qhi = __shfl_sync(kAll, my_hi, qi);
      }
    }
  };
  if (qi < 32) {
    qb = __shfl_sync(kAll, my_lo, qi);
    qhi = __shfl_sync(kAll, my_hi, qi);
    fetch(cur_u, cur_k);
    step_q();
    if (qi < 32) fetch(nxt_u, nxt_k);
    first(cur_u, cur_k);
  }
  for (int i = 0; i < nrows; ++i) {
    const Position lo = __shfl_sync(kAll, my_lo, i);
    const Position hi = __shfl_sync(kAll, my_hi, i);
    begin(here.x + i);
    for (Position b = lo; b < hi; b += 32) {
      batch(cur_u, cur_k, (int)b, (int)min(hi - b, 32u), nxt_u, nxt_k);
      cur_u = nxt_u;
      cur_k = nxt_k;
      if (qi < 32) {
        step_q();
        if (qi < 32) fetch(nxt_u, nxt_k);
      }
    }
    end(here.x + i, here.z);
  }
}
template <bool IDX, bool PERM, class Begin, class Batch, class End>
__device__ __forceinline__ void walk_chunk(const GenArgs& a, Begin begin, Batch batch, End end) {
  walk_chunk<IDX, PERM>(
      a, [](int32_t, int32_t) {}, begin,
      [&](int32_t u, int32_t k, int b, int cnt, int32_t, int32_t) { batch(u, k, b, cnt); }, end);
}

inline dim3 general_grid(const GenArgs& a, int vec) {
  const int per = (1 << a.log_g) * vec;
  return dim3((unsigned)((a.chunk_count + kGenWarps - 1) / kGenWarps),
              (unsigned)(a.slices ? a.slices : (a.F + per - 1) / per));
}

}  // namespace
#endif  // __CUDACC__
}  // namespace dg
#endif  // DG_GENERAL_CUH_
