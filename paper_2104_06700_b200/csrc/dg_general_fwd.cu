// Forward kernels of the general aggregation primitive, Eq. 1 of the paper for every operator pair of
// Table 1:  out[v][j] = (+) over the row of v of  x[colidx[k]][j] (x) y[k][j].
#include "dg_general.cuh"

namespace dg {
namespace {

// Bound by the gather like the sum kernels (copylhs, scalar edge operands), or by the stream of the edge
// features (full edge operand: nnz * F * 4 bytes, read once with streaming loads, which leave L2 to the
// gathered rows).  Six blocks per SM and four steps of loads in flight: three to eight blocks with two to
// eight steps were 0 to 60 % slower.  copylhs / max, B200: 31 M edges F = 100 2.41 -> 1.62 ms; 24 M edges
// F = 64 0.59 -> 0.51 ms; 5.7 M edges F = 602 (padded rows) 3.08 -> 1.15 ms.  mul / sum with full edge
// features, 7.9 M edges F = 64: 0.52 -> 0.34 ms (6.1 TB/s).
template <int BIN, int RED, int YM, int VEC, int U>
__global__ void __launch_bounds__(kGenBlock, 6) general_fwd_kernel(const GenArgs a) {
  const int lane = threadIdx.x & 31;
  const int G = 1 << a.log_g, NG = 32 >> a.log_g;
  const int grp = lane >> a.log_g, c = lane & (G - 1);
  const int f = (blockIdx.y + a.first_slice) * (G * VEC) + c * VEC;
  // lanes beyond F read the first features and never store: no load needs a predicate for them
  const float* xlane = a.X + (f < a.F ? f : 0);
  const float* ylane = a.Y + (f < a.F ? f : 0);
  float acc[VEC];    // the sum, or the extremum so far
  int32_t at[VEC];   // its edge position, -1: none
  bool fresh;        // the next step is the row's first

  auto step = [&](auto full, int32_t u, float ys, int b, int e0, int cnt) {
    constexpr bool kFullStep = decltype(full)::value;
    float x[U][VEC], y[U][VEC];
#pragma unroll
    for (int j = 0; j < U; ++j) {
      const int e = e0 + j * NG + grp;
      const bool valid = kFullStep || e < cnt;
#pragma unroll
      for (int q = 0; q < VEC; ++q) x[j][q] = y[j][q] = 0.f;
      if (BIN != kCopyRhs) {
        const int32_t id = __shfl_sync(kAll, u, e & 31);
        if (valid) load_vec<VEC>(x[j], xlane + (int64_t)id * a.ldx);
      }
      if (YM == kEdgeFull && valid) stream_vec<VEC>(y[j], ylane + (int64_t)(b + e) * a.F);
      if (YM == kEdgeScalar) {
        y[j][0] = __shfl_sync(kAll, ys, e & 31);
#pragma unroll
        for (int q = 1; q < VEC; ++q) y[j][q] = y[j][0];
      }
    }
#pragma unroll
    for (int j = 0; j < U; ++j) {
      const int e = e0 + j * NG + grp;
      const bool valid = kFullStep || e < cnt;
#pragma unroll
      for (int q = 0; q < VEC; ++q) {
        const float m = message<BIN>(x[j][q], y[j][q]);
        if (RED == kSum) {
          acc[q] += valid ? m : 0.f;
        } else {
          // A lane meets its edges in ascending position, so "strictly better" keeps the lowest
          // position among equal messages; lane groups and pieces are merged by take_better.  A lane
          // group that has edges in a row has the first of them in the row's first load step.
          const bool take = valid && ((j == 0 && fresh) || (RED == kMax ? m > acc[q] : m < acc[q]));
          acc[q] = take ? m : acc[q];
          at[q] = take ? b + e : at[q];
        }
      }
    }
    fresh = false;
  };

  walk_chunk<BIN != kCopyRhs, false>(
      a,
      [&](int) {
#pragma unroll
        for (int q = 0; q < VEC; ++q) {
          acc[q] = 0.f;
          at[q] = -1;
        }
        fresh = true;
      },
      [&](int32_t u, int32_t, int b, int cnt) {
        const float ys = (YM == kEdgeScalar && lane < cnt) ? __ldcs(a.Y + b + lane) : 0.f;
        int e0 = 0;
        for (; e0 + U * NG <= cnt; e0 += U * NG) step(True(), u, ys, b, e0, cnt);
        for (; e0 < cnt; e0 += U * NG) step(False(), u, ys, b, e0, cnt);
      },
      [&](int r, int slot) {
#pragma unroll
        for (int q = 0; q < VEC; ++q) {
          for (int off = G; off < 32; off <<= 1) {
            const float other = __shfl_xor_sync(kAll, acc[q], off);
            if (RED == kSum) {
              acc[q] += other;
            } else {
              take_better<RED>(acc[q], at[q], other, __shfl_xor_sync(kAll, at[q], off));
            }
          }
        }
        if (grp != 0 || f >= a.F) return;
        const int64_t o = (int64_t)(slot >= 0 ? slot : r) * a.F + f;
        float* out = slot >= 0 ? a.partial : a.out;
        int32_t* where = slot >= 0 ? a.partial_arg : a.arg_out;
#pragma unroll
        for (int q = 0; q < VEC; ++q) {
          if (f + q >= a.F) break;
          if (RED == kSum) {
            out[o + q] = a.accumulate ? out[o + q] + acc[q] : acc[q];
          } else {
            if (a.accumulate) take_better<RED>(acc[q], at[q], out[o + q], where[o + q]);
            out[o + q] = at[q] >= 0 ? acc[q] : 0.f;
            if (where) where[o + q] = at[q];
          }
        }
      });
}

// Merges the slots of every cut row into what the row's first chunk stored: thread per feature.
template <int RED>
__global__ void __launch_bounds__(128)
join_extrema_kernel(const Chunk* __restrict__ chunks, const CutRow* __restrict__ cuts,
                    const int32_t* __restrict__ totals, int32_t max_cuts, const float* __restrict__ partial,
                    const int32_t* __restrict__ partial_arg, int32_t F, float* __restrict__ out,
                    int32_t* __restrict__ arg_out) {
  const int f = blockIdx.y * 128 + threadIdx.x;
  const int cut_rows = min(__ldg(totals + 1), max_cuts);
  if (f >= F) return;
  for (int i = blockIdx.x; i < cut_rows; i += gridDim.x) {
    const CutRow cut = cuts[i];
    const int64_t o = (int64_t)cut.row * F + f;
    float best = out[o];
    // without arg the pieces' order decides ties: the first piece of a row is never empty then
    int32_t at = arg_out ? arg_out[o] : 0;
#pragma unroll 4
    for (int k = 0; k < cut.count; ++k) {
      const int64_t p = (int64_t)__ldg(&chunks[cut.first + k].slot) * F + f;
      const float m = partial[p];
      const int32_t mk = partial_arg[p];
      if (arg_out) take_better<RED>(best, at, m, mk);
      else if (mk >= 0 && (RED == kMax ? m > best : m < best)) best = m;
    }
    out[o] = best;
    if (arg_out) arg_out[o] = at;
  }
}

template <int BIN, int RED, int YM, int VEC>
dg_status_t launch(const GenArgs& a, cudaStream_t s) {
  const dim3 grid = general_grid(a, VEC);
  // a batch has 32 edges, which narrow groups cover in fewer steps
  if (a.log_g >= 3) general_fwd_kernel<BIN, RED, YM, VEC, 4><<<grid, kGenBlock, 0, s>>>(a);
  else general_fwd_kernel<BIN, RED, YM, VEC, 2><<<grid, kGenBlock, 0, s>>>(a);
  DG_CUDA(cudaGetLastError());
  count_launches(1);
  return DG_OK;
}

template <int BIN, int RED>
dg_status_t by_edge_operand(const GenArgs& a, cudaStream_t s) {
  if constexpr (BIN != kCopyLhs) {
    if (a.cols != 1) {
      if (a.vec == 4) return launch<BIN, RED, kEdgeFull, 4>(a, s);
      if (a.vec == 2) return launch<BIN, RED, kEdgeFull, 2>(a, s);
      return launch<BIN, RED, kEdgeFull, 1>(a, s);
    }
  }
  constexpr int YM = BIN == kCopyLhs ? kNoEdge : kEdgeScalar;
  if (a.vec == 4) return launch<BIN, RED, YM, 4>(a, s);
  if (a.vec == 2) return launch<BIN, RED, YM, 2>(a, s);
  return launch<BIN, RED, YM, 1>(a, s);
}

template <int BIN>
dg_status_t by_reducer(const GenArgs& a, int red, cudaStream_t s) {
  if (red == kMax) return by_edge_operand<BIN, kMax>(a, s);
  if (red == kMin) return by_edge_operand<BIN, kMin>(a, s);
  if constexpr (BIN == kCopyLhs) return DG_ERR_UNSUPPORTED;  // dg_ap_fwd hands it to aggregate_sum
  else return by_edge_operand<BIN, kSum>(a, s);
}

}  // namespace

dg_status_t launch_general_fwd(const GenArgs& a, int bin, int red, cudaStream_t s) {
  switch (bin) {
    case kCopyLhs: return by_reducer<kCopyLhs>(a, red, s);
    case kCopyRhs: return by_reducer<kCopyRhs>(a, red, s);
    case kAdd: return by_reducer<kAdd>(a, red, s);
    case kSub: return by_reducer<kSub>(a, red, s);
    case kMul: return by_reducer<kMul>(a, red, s);
    default: return by_reducer<kDiv>(a, red, s);
  }
}

dg_status_t join_extrema(const Graph* g, const Plan& plan, const GenArgs& a, int red, cudaStream_t s) {
  // the number of cut rows may still be on its way to the host: the kernel reads it on the device
  int64_t blocks = plan.cut_rows >= 0 ? plan.cut_rows : plan.max_cuts;
  if (blocks > (int64_t)g->sm_count * 64) blocks = (int64_t)g->sm_count * 64;
  const dim3 grid((unsigned)blocks, (unsigned)((a.F + 127) / 128));
  if (red == kMax)
    join_extrema_kernel<kMax><<<grid, 128, 0, s>>>(plan.chunks, plan.cuts, plan.totals, (int32_t)plan.max_cuts,
                                                   a.partial, a.partial_arg, a.F, a.out, a.arg_out);
  else
    join_extrema_kernel<kMin><<<grid, 128, 0, s>>>(plan.chunks, plan.cuts, plan.totals, (int32_t)plan.max_cuts,
                                                   a.partial, a.partial_arg, a.F, a.out, a.arg_out);
  DG_CUDA(cudaGetLastError());
  count_launches(1);
  return DG_OK;
}

}  // namespace dg
