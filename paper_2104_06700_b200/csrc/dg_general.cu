// The general aggregation primitive: every operator pair of Table 1 of the paper,
//   f_O[v] = (+)_{edges e_uv into v} ( f_V[u] (x) f_E[e_uv] )          (Eq. 1, Eq. 2, Algorithm 1)
// with (x) in {copylhs, copyrhs, add, sub, mul, div}, (+) in {sum, max, min} and f_E a full
// |E| x F matrix (or |E| x 1, broadcast), its gradients with respect to f_V and f_E, and the
// gradient of the weighted sum / mean with respect to scalar edge weights (message passing onto
// edges, Section 2.2).  This file checks arguments and chooses launches; the kernels are in
// dg_general_fwd.cu, dg_general_bwd.cu and dg_edge_grad.cu (the units compile side by side).
#include "dg_general.cuh"

namespace dg {
namespace {

int log_group(int32_t width) {  // lanes per edge: the power of two covering `width`, at most 32
  int lg = 0;
  while (lg < 5 && (1 << lg) < width) ++lg;
  return lg;
}

// Source blocks of one general call, like the sum / mean kernels' (Algorithm 2 with L2 as the cache): when
// the gathered matrices (`row_bytes` of them for one slice of 128 features) do not fit the handle's L2
// budget, the call runs as one launch per range of neighbour ids and slice of features; the ranges
// partition the edges and each launch folds its piece into the output of the earlier
// ones (can_merge: max / min need the arg matrix for that).  Without split pointers, or where the pieces
// of a row would fall under 32 edges, the call stays one launch.  The handle's "source_blocks" attribute
// forces the number of ranges.
int plan_blocks(const dg_graph* g, double row_bytes, const int32_t* split, bool can_merge) {
  if (!split || !can_merge || row_bytes == 0.0) return 1;
  if (g->source_blocks > 0) return (int)g->source_blocks;
  const double budget = (double)g->l2_budget_bytes;
  int nb = 1;
  while (nb < kFineBlocks && (double)g->n / nb * row_bytes > budget) nb *= 2;
  return (double)g->nnz / (double)g->n / nb >= 32.0 ? nb : 1;
}

// bytes a slice of up to 128 floats occupies in L2, where it rarely starts on a line
double slice_bytes(int64_t F) {
  const int64_t w = F < 128 ? F : 128;
  return (double)(w * 4 + (F > w ? 128 : 0));
}

void use_plan(const dg_graph* g, bool over_csc, GenArgs* a) {
  const Plan& plan = over_csc ? g->col_plan : g->row_plan;
  a->chunks = plan.chunks;
  a->chunk_count = (int32_t)plan.count;
  a->ptr = over_csc ? g->colptr : g->rowptr;
  a->idx = over_csc ? g->rowidx_T : g->colidx;
  a->perm = over_csc ? g->perm : nullptr;
}

// One launch per range of neighbour ids and slice of per_lane << log_g features (all slices in one grid
// when there is one range); the parts of cut rows go to a.partial.
template <class Launch>
dg_status_t run_blocks(const dg_graph* g, GenArgs a, const int32_t* split, int nb, int per_lane, Launch launch) {
  const int per = kFineBlocks / nb;
  dg_status_t st = DG_OK;
  for (int j = 0; j < nb && st == DG_OK; ++j) {
    if (nb > 1) {
      a.seg_lo = split + (size_t)(j * per) * (size_t)g->n;
      a.seg_hi = split + (size_t)((j + 1) * per) * (size_t)g->n;
    }
    a.accumulate = j > 0;
    if (nb == 1 || per_lane == 0) {
      st = launch(a);
      continue;
    }
    a.slices = 1;
    for (a.first_slice = 0; a.first_slice * (per_lane << a.log_g) < a.F && st == DG_OK; ++a.first_slice)
      st = launch(a);
  }
  return st;
}

int vector_width(int32_t F, uintptr_t pointers) {
  return (F % 4 == 0 && (pointers & 15) == 0) ? 4 : (F % 2 == 0 && (pointers & 7) == 0) ? 2 : 1;
}

// 16-byte loads of a gathered matrix whose rows forbid them, through a padded copy (*copy: for pool_free)
dg_status_t widen(const dg_graph* g, GenArgs* a, cudaStream_t s, void** copy) {
  if (!worth_padding(g, a->F, 4, a->vec)) return DG_OK;
  if (dg_status_t st = pad_rows(g, a->X, a->F, 4, nullptr, 0, s, copy, &a->ldx)) return st;
  if (*copy) {
    a->X = static_cast<const float*>(*copy);
    a->vec = 4;
  }
  return DG_OK;
}

// dV of max / min.  The mask of the selected edges (see dg_general_bwd.cu) is made and used for up to 256
// features at a time, as many as fit kMaskMaxBytes: one 32-byte sector per edge holds 256 bits.
constexpr size_t kMaskMaxBytes = (size_t)2 << 30;  // the pool keeps this much

// Whether dV of max / min goes through the mask, or compares arg edge by edge.  The mask saves gathered rows but costs a
// launch, scratch and a pass over the rows, so calls on fewer than kMaskMinEdges compare, unless
// rows are short (124 k edges in rows of 4, F = 4: 18.5 / 20.6 us); and for 9 to 16 features its kernel has 16 lanes per
// edge where the comparison has four.  The factors of mul / div make the comparison dearer.
// Measured, us with / without the mask, copylhs: 57 k edges F = 16 18.5 / 9.5, F = 128 24.7 / 20.7; 158 k F = 64 20.6 /
// 13.0, F = 602 92 / 86; 573 k F = 8 23.5 / 22.6, F = 32 36 / 27, F = 100 55 / 59; F = 16 at mean degree 4 309 / 458, 14.5
// 732 / 714, 50 148 / 122, 110 125 / 92, 270 576 / 406.  mul with one column: 57 k F = 16 18.5 / 12.3, F = 64 22.6 / 26.7;
// F = 16 at mean degree 14.5 908 / 1098, 50 962 / 1048, 84 49 / 38, 270 726 / 648.
constexpr int64_t kMaskMinEdges = 1 << 17;
bool mask_pays(const dg_graph* g, int32_t F, int32_t cols, int bin) {
  const bool factors = bin == kMul || bin == kDiv;
  if (factors && cols != 1) return true;
  if (g->nnz < kMaskMinEdges) return g->nnz < 8 * g->n || (factors && F > 32);
  return F <= 8 || F > 16 || g->nnz < (factors ? 64 : 24) * g->n;
}
dg_status_t extremum_dv(const dg_graph* g, GenArgs a, int bin, int red, cudaStream_t s) {
  const int blocks = g->split_csc && g->source_blocks > 1 ? (int)g->source_blocks : 1;
  int words = 1;
  while (words < (blocks > 1 ? 4 : 8) && words * 32 < a.F) words *= 2;
  while (words > 1 && (size_t)g->nnz * (size_t)words * 4 > kMaskMaxBytes) words /= 2;
  void* mask = nullptr;
  auto dv = [&](const GenArgs& p) { return launch_general_dv(p, bin, red, s); };
  if (g->nnz == 0 || !mask_pays(g, a.F, a.cols, bin) || (size_t)g->nnz * (size_t)words * 4 > kMaskMaxBytes ||
      scratch_alloc(g, (size_t)g->nnz * (size_t)words * 4, s, &mask) != cudaSuccess) {
    a.vec = vector_width(a.F, (uintptr_t)a.arg) == 4 ? 4 : 1;  // of arg; a lane has four features
    a.log_g = log_group((a.F + 3) / 4);
    const int nb = plan_blocks(g, 2 * slice_bytes(a.F), g->split_csc, true);  // dO and arg
    return run_blocks(g, a, g->split_csc, nb, 4, dv);
  }
  a.mask = static_cast<uint32_t*>(mask);
  a.log_g = log_group(a.F);
  GenArgs rows = a;
  use_plan(g, false, &rows);
  dg_status_t st = DG_OK;
  for (int f0 = 0; f0 < a.F && st == DG_OK; f0 += 32 * words) {
    while (words > 1 && a.F - f0 <= 16 * words) words /= 2;  // what is left
    a.f_lo = rows.f_lo = f0;
    a.words = rows.words = words;
    st = launch_arg_mask(rows, s);
    // the selected values of dO are too few for L2 to matter: source blocks only on request
    if (st == DG_OK) st = run_blocks(g, a, g->split_csc, blocks, 0, dv);
  }
  pool_free(mask, s);
  return st;
}

// The later pieces of a call that found no memory for their results.
PieceArgs pieces_of(const GenArgs& a, int bin, int red, bool gradient) {
  PieceArgs p{};
  p.idx = bin == kCopyRhs ? nullptr : a.idx;
  p.perm = a.perm;
  p.X = a.X;
  p.ldx = a.ldx;
  p.Y = bin == kCopyLhs ? nullptr : a.Y;
  p.edge_cols = a.cols;
  p.arg = a.arg;
  p.F = a.F;
  p.bin = bin;
  p.red = red;
  p.gradient = gradient;
  p.out = a.out;
  p.arg_out = a.arg_out;
  return p;
}

dg_status_t bad(const char* msg) {
  set_error("%s", msg);
  return DG_ERR_INVALID_ARG;
}

dg_status_t check_operands(const dg_graph* g, const float* fV, const float* fE, int32_t fE_cols,
                           int32_t F, int bin, int red) {
  if (!g) return bad("graph handle is NULL");
  if (F < 1) return bad("F must be >= 1");
  if (F > (1 << 20)) {
    set_error("F must be at most 2^20");
    return DG_ERR_UNSUPPORTED;
  }
  if (bin < kCopyLhs || bin > kDiv) return bad("binary must be one of the dg_binary_t values");
  if (red < kSum || red > kMin) return bad("reduce must be one of the dg_reduce_t values");
  if (bin != kCopyRhs && !fV && g->n > 0) return bad("fV is NULL (only copyrhs works without it)");
  if (bin != kCopyLhs) {
    if (!fE && g->nnz > 0) return bad("fE is NULL (only copylhs works without it)");
    if (fE_cols != 1 && fE_cols != F) return bad("fE_cols must be 1 or F");
  }
  return DG_OK;
}

}  // namespace
}  // namespace dg

using namespace dg;

extern "C" {

dg_status_t dg_ap_fwd(dg_graph_t g, const float* fV, const float* fE, int32_t fE_cols, int32_t F,
                      dg_binary_t binary, dg_reduce_t reduce, float* fO, int32_t* arg,
                      void* stream) {
  if (dg_status_t st = check_operands(g, fV, fE, fE_cols, F, (int)binary, (int)reduce)) return st;
  if (g->n == 0) return DG_OK;
  if (!fO) return bad("fO is NULL");
  // copylhs / sum is the plain sum, mul / sum with one column the weighted sum with fE as the
  // weights: the sum / mean kernels do these two (about 2.5x faster on the dense graphs)
  if (reduce == DG_RED_SUM &&
      (binary == DG_BIN_COPY_LHS || (binary == DG_BIN_MUL && fE_cols == 1)))
    return aggregate_sum(g, false, binary == DG_BIN_MUL ? fE : nullptr, fV, F, fO,
                         (cudaStream_t)stream);
  cudaStream_t s = (cudaStream_t)stream;
  const bool extremum = reduce != DG_RED_SUM;
  GenArgs a{};
  use_plan(g, false, &a);
  a.X = fV;
  a.ldx = F;
  a.Y = fE;
  a.out = fO;
  a.arg_out = extremum ? arg : nullptr;
  a.F = F;
  a.cols = binary == DG_BIN_COPY_LHS ? 1 : fE_cols;
  // the rows that are loaded as vectors: fV's (none for copyrhs), and fE's when it has F columns
  const uintptr_t rows = (binary == DG_BIN_COPY_RHS ? 0 : (uintptr_t)fV) | (a.cols != 1 ? (uintptr_t)fE : 0);
  a.vec = vector_width(F, rows);
  void* padded = nullptr;
  if (a.cols == 1 && binary != DG_BIN_COPY_RHS)
    if (dg_status_t st = widen(g, &a, s, &padded)) return st;
  a.log_g = log_group((F + a.vec - 1) / a.vec);
  // copyrhs gathers nothing: its edge rows are a stream
  const int nb = plan_blocks(g, binary == DG_BIN_COPY_RHS ? 0.0 : slice_bytes(a.ldx), g->split_csr,
                             !extremum || arg != nullptr);
  // an extremum's parts carry their edge positions
  const Plan& plan = g->row_plan;
  bool missing = false;
  a.partial = take_partial(g, plan, (int64_t)F * (extremum ? 2 : 1), s, &missing);
  a.skip_pieces = missing;
  if (extremum && a.partial)
    a.partial_arg =
        reinterpret_cast<int32_t*>(a.partial + (plan.slots >= 0 ? plan.slots : plan.max_slots) * (int64_t)F);
  dg_status_t st = run_blocks(g, a, g->split_csr, nb, a.vec, [&](const GenArgs& p) {
    return launch_general_fwd(p, (int)binary, (int)reduce, s);
  });
  if (missing && st == DG_OK) st = add_pieces(g, plan, pieces_of(a, (int)binary, (int)reduce, false), s);
  if (a.partial) {
    if (st == DG_OK)
      st = extremum ? join_extrema(g, plan, a, (int)reduce, s) : join_cut_rows(g, plan, a.partial, F, fO, s);
    pool_free(a.partial, s);
  }
  pool_free(padded, s);
  return st;
}

dg_status_t dg_ap_bwd(dg_graph_t g, const float* dO, const float* fV, const float* fE,
                      int32_t fE_cols, int32_t F, dg_binary_t binary, dg_reduce_t reduce,
                      const int32_t* arg, float* dV, float* dE, void* stream) {
  if (dg_status_t st = check_operands(g, fV, fE, fE_cols, F, (int)binary, (int)reduce)) return st;
  if (g->n == 0) return DG_OK;
  if (!dO) return bad("dO is NULL");
  if (reduce != DG_RED_SUM && !arg) return bad("max / min need the arg output of dg_ap_fwd");
  if (dE && binary == DG_BIN_COPY_LHS) return bad("copylhs has no edge operand: dE must be NULL");
  cudaStream_t s = (cudaStream_t)stream;
  const int32_t cols = binary == DG_BIN_COPY_LHS ? 1 : fE_cols;
  if (dV) {
    if (binary == DG_BIN_COPY_RHS) {  // the result does not depend on fV
      DG_CUDA(cudaMemsetAsync(dV, 0, (size_t)g->n * (size_t)F * sizeof(float), s));
    } else {
      if (!g->transposed) {
        set_error("the gradient with respect to fV gathers over the CSC: call dg_graph_transpose first");
        return DG_ERR_NOT_TRANSPOSED;
      }
      // sum with copylhs / add / sub: dV[u] is the plain sum of dO over the out-edges of u
      if (reduce == DG_RED_SUM && (binary == DG_BIN_COPY_LHS || binary == DG_BIN_ADD ||
                                   binary == DG_BIN_SUB)) {
        if (dg_status_t st = aggregate_sum(g, true, nullptr, dO, F, dV, s)) return st;
      } else {
        GenArgs a{};
        use_plan(g, true, &a);
        a.X = dO;
        a.ldx = F;
        a.Y = fE;
        a.arg = arg;
        a.out = dV;
        a.F = F;
        a.cols = cols;
        const Plan& plan = column_plan(g);
        bool missing = false;
        a.partial = take_partial(g, plan, F, s, &missing);
        a.skip_pieces = missing;
        dg_status_t st = DG_OK;
        if (reduce != DG_RED_SUM) {
          st = extremum_dv(g, a, (int)binary, (int)reduce, s);
          if (missing && st == DG_OK) st = add_pieces(g, plan, pieces_of(a, (int)binary, (int)reduce, true), s);
        } else {
          a.vec = vector_width(F, (uintptr_t)dO | (cols != 1 ? (uintptr_t)fE : 0));
          void* padded = nullptr;
          if (cols == 1) st = widen(g, &a, s, &padded);
          a.log_g = log_group((F + a.vec - 1) / a.vec);
          const int nb = plan_blocks(g, slice_bytes(a.ldx), g->split_csc, true);
          if (st == DG_OK)
            st = run_blocks(g, a, g->split_csc, nb, a.vec,
                            [&](const GenArgs& p) { return launch_general_dv(p, (int)binary, (int)reduce, s); });
          if (missing && st == DG_OK) st = add_pieces(g, plan, pieces_of(a, (int)binary, (int)reduce, true), s);
          pool_free(padded, s);
        }
        if (a.partial) {
          if (st == DG_OK) st = join_cut_rows(g, plan, a.partial, F, dV, s);
          pool_free(a.partial, s);
        }
        if (st != DG_OK) return st;
      }
    }
  }
  if (dE && g->nnz > 0) {
    // mul / sum with one edge column: dE[k] = <fV[u_k], dO[v_k]>, the edge-weight gradient of the sum
    if (binary == DG_BIN_MUL && reduce == DG_RED_SUM && cols == 1)
      return dg_aggregate_edge_grad(g, fV, dO, F, DG_OP_SUM, dE, stream);
    GenArgs a{};
    use_plan(g, false, &a);
    a.X = dO;
    a.V = fV;
    a.Y = fE;
    a.arg = arg;
    a.out = dE;
    a.F = F;
    a.cols = cols;
    a.vec = 1;
    if (cols != 1) {  // 16-byte rows of every matrix the full-width kernel touches
      uintptr_t all = (uintptr_t)dO | (uintptr_t)dE;
      if (binary == DG_BIN_MUL || binary == DG_BIN_DIV) all |= (uintptr_t)fV;
      if (binary == DG_BIN_DIV) all |= (uintptr_t)fE;
      if (reduce != DG_RED_SUM) all |= (uintptr_t)arg;
      if (vector_width(F, all) == 4) a.vec = 4;
    }
    a.log_g = log_group((F + a.vec - 1) / a.vec);
    return launch_general_de(a, (int)binary, (int)reduce, s);
  }
  return DG_OK;
}

dg_status_t dg_aggregate_edge_grad(dg_graph_t g, const float* H, const float* dOut, int32_t F,
                                   dg_op_t op, float* dW, void* stream) {
  if (!g) return bad("graph handle is NULL");
  if (F < 1) return bad("F must be >= 1");
  if (F > (1 << 20)) {
    set_error("F must be at most 2^20");
    return DG_ERR_UNSUPPORTED;
  }
  if (op != DG_OP_SUM && op != DG_OP_MEAN) return bad("op must be DG_OP_SUM or DG_OP_MEAN");
  if (g->nnz == 0) return DG_OK;
  if (!H || !dOut || !dW) return bad("H, dOut or dW is NULL");
  return edge_grad_run(g, H, dOut, F, op == DG_OP_MEAN ? (g->self_loops ? 2 : 1) : 0, dW,
                       (cudaStream_t)stream);
}

}  // extern "C"
