// dg_aggregate_edge_grad: dW[k] = s_v * <H[u_k], dOut[v_k]>, one dot product per edge (message passing
// onto edges, Section 2.2 of the paper).
//
// A warp takes one chunk of the CSR's plan.  G lanes take one edge, VEC floats per lane and load, U edges
// are in flight per lane group before the first multiply.  dOut[v] is the same row for every edge of v: a
// slab of it is read (from L1) once per U edges.  The U partial dot products of a group are reduced
// together by a transposing butterfly: U - 1 + log2(G / U) shuffles instead of U * log2(G).
// Bound like the forward pass by the gathered rows of H: 39.6 M edges, F = 64 1.12 -> 0.78 ms (13 TB/s
// gathered from L2; the shuffles and the second operand are what is left over the sum's 0.53).
#include "dg_general.cuh"

namespace dg {
namespace {

struct EdgeGradArgs {
  GenArgs walk;       // chunks, pointers, ids, pieces of a source-blocked launch
  const float* H;
  const float* dOut;
  int64_t ld;         // floats between rows of H and dOut
  float* dW;
  int32_t row_scale;  // 0 none, 1 = 1/deg(v), 2 = 1/(deg(v)+1)
  int32_t f_lo, nvec; // the launch's slice: nvec vectors from feature f_lo on
  int32_t accumulate; // dW already holds the dot products of the earlier feature slices
};

template <int VEC> struct LoadVec;
template <> struct LoadVec<1> { using T = float; };
template <> struct LoadVec<2> { using T = float2; };
template <> struct LoadVec<4> { using T = float4; };
__device__ __forceinline__ float dotv(float x, float g) { return x * g; }
__device__ __forceinline__ float dotv(float2 x, float2 g) { return x.x * g.x + x.y * g.y; }
__device__ __forceinline__ float dotv(float4 x, float4 g) {
  return x.x * g.x + x.y * g.y + x.z * g.z + x.w * g.w;
}

// four blocks per SM (64 registers): U loads of 16 bytes stay in flight
template <int VEC, int G>
__global__ void __launch_bounds__(kGenBlock, 4) edge_grad_kernel(const EdgeGradArgs a) {
  using V = typename LoadVec<VEC>::T;
  constexpr int U = G < 8 ? G : 8;  // edges per lane group: 32 / G groups * U edges <= a batch of 32
  const int lane = threadIdx.x & 31;
  const int grp = lane / G, c = lane % G;
  const V* grow = nullptr;
  float s = 1.f;
  walk_chunk<true, false>(
      a.walk,
      [&](int v) {
        grow = reinterpret_cast<const V*>(a.dOut + (int64_t)v * a.ld + a.f_lo);
        if (a.row_scale)
          s = 1.0f / (float)(__ldg(a.walk.ptr + v + 1) - __ldg(a.walk.ptr + v) + (a.row_scale == 2 ? 1 : 0));
      },
      [&](int32_t my_u, int32_t, int b, int cnt) {
        for (int e0 = 0; e0 < cnt; e0 += U * (32 / G)) {
          // the group's edges are e0 + grp * U + j; lanes past the batch name vertex 0: their loads are
          // harmless and never written
          const V* xrow[U];
          float p[U];
#pragma unroll
          for (int j = 0; j < U; ++j) {
            const int32_t u = __shfl_sync(kAll, my_u, (e0 + grp * U + j) & 31);
            xrow[j] = reinterpret_cast<const V*>(a.H + (int64_t)u * a.ld + a.f_lo);
            p[j] = 0.f;
          }
          for (int t = c; t < a.nvec; t += G) {
            const V gt = __ldg(grow + t);
            V x[U];
#pragma unroll
            for (int j = 0; j < U; ++j) x[j] = __ldg(xrow[j] + t);
#pragma unroll
            for (int j = 0; j < U; ++j) p[j] += dotv(x[j], gt);
          }
          // Exchange steps halve the number of sums a lane holds (lanes with the step's bit set keep the
          // upper half); when one is left, the remaining steps only add.
          int held = U, first = 0;
#pragma unroll
          for (int off = G / 2; off >= 1; off >>= 1) {
            const bool up = lane & off;
            if (held > 1) {
              held /= 2;
#pragma unroll
              for (int i = 0; i < U / 2; ++i) {
                if (i < held) {
                  const float got = __shfl_xor_sync(kAll, up ? p[i] : p[i + held], off);
                  p[i] = (up ? p[i + held] : p[i]) + got;
                }
              }
              if (up) first += held;
            } else {
              p[0] += __shfl_xor_sync(kAll, p[0], off);
            }
          }
          const int e = e0 + grp * U + first;
          if ((c & (G / U - 1)) == 0 && e < cnt) {
            float* w = a.dW + b + e;
            *w = a.accumulate ? *w + p[0] * s : p[0] * s;
          }
        }
      },
      [](int, int) {});
}

// Lanes per edge.  Lanes for all vectors up to 32, or half of those: a lane then takes two vectors of a row, and the shuffles
// (an id per edge and load, and the butterfly), which share a pipe with the loads, serve twice the loads.  us with all / half,
// rows of 422 entries (L2), of 50 (376 MB), of 14.5 (306 MB and less):
//    4 vectors   456 / 386   1626 / 1324   188 / 159; two lanes 380   1233   137: two lanes, for every length
//    5           458 / 636   1762 / 2014   196 / 261: up to 8 otherwise all
//   12           779 / 617   2839 / 2802   255 / 303: from 9 on half where a row has edges for the groups, 32
//   16           774 / 628   2825 / 3011   254 / 324: 13 to 16 only where L2 keeps the matrix (36 entries, 77 MB: 325 / 335)
//   32          1399 / 1139  5009 / 4866   360 / 386
// Half of that again where fewer lanes are then without a vector: 12 vectors (four lanes 632, 2505), 20 (eight lanes 805,
// 4115 against 1070, 4349), and for every length 43 (16 lanes against 32: 1649 / 2149, 7508 / 8509, 537 / 546).
int lanes_per_edge(int nvec, double entries, bool resident) {
  if (nvec == 4) return 2;
  int lanes = 1;
  while (lanes < 32 && lanes < nvec) lanes *= 2;
  const bool half = entries >= 32.0 && nvec > 8 && (resident || nvec <= 12 || nvec > 16);
  if (half && nvec <= 32) lanes /= 2;
  auto slots = [&](int l) { return (nvec + l - 1) / l * l; };
  if ((half || nvec > 32) && nvec <= 2 * lanes && slots(lanes / 2) < slots(lanes)) lanes /= 2;
  return lanes;
}

template <int VEC, int G>
dg_status_t launch_lanes(const EdgeGradArgs& a, cudaStream_t s) {
  edge_grad_kernel<VEC, G><<<(unsigned)((a.walk.chunk_count + kGenWarps - 1) / kGenWarps), kGenBlock, 0, s>>>(a);
  DG_CUDA(cudaGetLastError());
  count_launches(1);
  return DG_OK;
}

template <int VEC>
dg_status_t launch_edge_grad(const EdgeGradArgs& a, double entries, bool resident, cudaStream_t s) {
  switch (lanes_per_edge(a.nvec, entries, resident)) {
    case 1: return launch_lanes<VEC, 1>(a, s);
    case 2: return launch_lanes<VEC, 2>(a, s);
    case 4: return launch_lanes<VEC, 4>(a, s);
    case 8: return launch_lanes<VEC, 8>(a, s);
    case 16: return launch_lanes<VEC, 16>(a, s);
    default: return launch_lanes<VEC, 32>(a, s);
  }
}

}  // namespace

dg_status_t edge_grad_run(const Graph* g, const float* H, const float* dOut, int32_t F, int row_scale,
                          float* dW, cudaStream_t s) {
  EdgeGradArgs a{};
  a.walk.chunks = g->row_plan.chunks;
  a.walk.chunk_count = (int32_t)g->row_plan.count;
  a.walk.ptr = g->rowptr;
  a.walk.idx = g->colidx;
  a.H = H;
  a.dOut = dOut;
  a.dW = dW;
  a.ld = F;
  a.row_scale = row_scale;
  const uintptr_t both = (uintptr_t)H | (uintptr_t)dOut;
  int vec = (F % 4 == 0 && (both & 15) == 0) ? 4 : (F % 2 == 0 && (both & 7) == 0) ? 2 : 1;
  void *padded_h = nullptr, *padded_g = nullptr;
  dg_status_t st = DG_OK;
  if (worth_padding(g, F, 4, vec)) {
    // both rows of a dot product in the same padded layout; the padding multiplies to zero
    int64_t ld = 0;
    st = pad_rows(g, H, F, 4, nullptr, 0, s, &padded_h, &ld);
    if (st == DG_OK && padded_h) st = pad_rows(g, dOut, F, 4, nullptr, 0, s, &padded_g, &ld);
    if (padded_h && padded_g) {
      a.H = static_cast<const float*>(padded_h);
      a.dOut = static_cast<const float*>(padded_g);
      a.ld = ld;
      vec = 4;
    }
  }
  // Like the aggregation itself (Algorithm 2 with L2 as the cache): when the gathered matrix does not stay
  // L2-resident and the rows carry split pointers, the call is cut into feature slices and source-vertex
  // blocks sized to the L2 budget, one launch each; the blocks partition the edges, the slices add up in
  // dW (each reads and writes it again: the widest slice whose blocks leave 32 edges of a row is taken).
  const int64_t width = (F + vec - 1) / vec * vec;
  int64_t slice = width;
  int nb = 1;
  if (g->split_csr && (double)g->n * (double)a.ld * 4.0 > (double)g->l2_budget_bytes) {
    for (int64_t w = 128LL * vec; w >= 32LL * vec; w /= 2) {
      const int64_t cand = w < width ? w : width;
      int blocks = 1;
      while (blocks < kFineBlocks &&
             (double)g->n / blocks * (double)(cand * 4 + 128) > (double)g->l2_budget_bytes)
        blocks *= 2;
      if ((double)g->nnz / (double)g->n / blocks < 32.0) continue;  // pieces too short to pay
      slice = cand;
      nb = blocks;
      break;
    }
  }
  const int per = kFineBlocks / nb;
  const double entries = (double)g->nnz / (double)g->n / nb; // of a row, in a launch
  const bool resident = nb > 1 || (double)g->n * (double)a.ld * 4.0 <= (double)g->l2_budget_bytes;
  for (int j = 0; j < nb && st == DG_OK; ++j) {
    if (nb > 1) {
      a.walk.seg_lo = g->split_csr + (size_t)(j * per) * (size_t)g->n;
      a.walk.seg_hi = g->split_csr + (size_t)((j + 1) * per) * (size_t)g->n;
    }
    for (int64_t f0 = 0; f0 < width && st == DG_OK; f0 += slice) {
      a.f_lo = (int32_t)f0;
      a.nvec = (int32_t)((width - f0 < slice ? width - f0 : slice) / vec);
      a.accumulate = f0 > 0;
      st = vec == 4   ? launch_edge_grad<4>(a, entries, resident, s)
           : vec == 2 ? launch_edge_grad<2>(a, entries, resident, s)
                      : launch_edge_grad<1>(a, entries, resident, s);
    }
  }
  pool_free(padded_h, s);
  pool_free(padded_g, s);
  return st;
}

}  // namespace dg
