// Gradients of the general aggregation primitive.  With sel = 1 for sum and [arg[v][j] == k] for max / min:
//   dV[u][j] = sum over the CSC column of u of  sel * dO[v][j] * d(x (x) y)/dx
//   dE[k][j] =                                  sel * dO[v][j] * d(x (x) y)/dy
// (dE summed over j when fE has one column).
#include "dg_general.cuh"

namespace dg {
namespace {

// Sums over the lane groups and stores one row (or part of a cut row) of dV: lane c of a group holds the
// features f, f + step, f + 2 step, ...
template <int N>
__device__ __forceinline__ void store_sum(const GenArgs& a, float (&acc)[N], int r, int slot, int f, int step,
                                          int G, int grp) {
#pragma unroll
  for (int q = 0; q < N; ++q)
    for (int off = G; off < 32; off <<= 1) acc[q] += __shfl_xor_sync(kAll, acc[q], off);
  if (grp != 0) return;
  float* o = (slot >= 0 ? a.partial : a.out) + (int64_t)(slot >= 0 ? slot : r) * a.F;
#pragma unroll
  for (int q = 0; q < N; ++q) {
    const int fq = f + q * step;
    if (fq < a.F) o[fq] = a.accumulate ? o[fq] + acc[q] : acc[q];
  }
}

// dV of mul / div under sum (with copylhs, add and sub it is the plain sum of dO): per edge the row dO[v]
// and the row (or scalar) fE[k] at the edge's CSR position, which are random rows in the CSC's order.
// Bound by HBM when fE is full, nnz rows of F floats: 7.9 M edges, F = 64 0.62 -> 0.36 ms (6 TB/s).
template <int BIN, int YM, int VEC, int U>
__global__ void __launch_bounds__(kGenBlock, 4) general_dv_sum_kernel(const GenArgs a) {
  const int lane = threadIdx.x & 31;
  const int G = 1 << a.log_g, NG = 32 >> a.log_g;
  const int grp = lane >> a.log_g, c = lane & (G - 1);
  const int f = (blockIdx.y + a.first_slice) * (G * VEC) + c * VEC;
  const float* xlane = a.X + (f < a.F ? f : 0);
  const float* ylane = a.Y + (f < a.F ? f : 0);
  float acc[VEC];

  auto step = [&](auto full, int32_t v, int32_t k, float ys, int e0, int cnt) {
    constexpr bool kFullStep = decltype(full)::value;
    float x[U][VEC], y[U][VEC];
#pragma unroll
    for (int j = 0; j < U; ++j) {
      const int e = e0 + j * NG + grp;
      const bool valid = kFullStep || e < cnt;
#pragma unroll
      for (int q = 0; q < VEC; ++q) {
        x[j][q] = 0.f;
        y[j][q] = BIN == kDiv ? 1.f : 0.f;  // absent edges: a division by zero takes a slow path
      }
      const int32_t id = __shfl_sync(kAll, v, e & 31);
      if (valid) load_vec<VEC>(x[j], xlane + (int64_t)id * a.ldx);
      if (YM == kEdgeFull) {
        const int32_t pos = __shfl_sync(kAll, k, e & 31);
        if (valid) stream_vec<VEC>(y[j], ylane + (int64_t)pos * a.F);
      } else {
        y[j][0] = __shfl_sync(kAll, ys, e & 31);
#pragma unroll
        for (int q = 1; q < VEC; ++q) y[j][q] = y[j][0];
      }
    }
#pragma unroll
    for (int j = 0; j < U; ++j) {
      const bool valid = kFullStep || e0 + j * NG + grp < cnt;
#pragma unroll
      for (int q = 0; q < VEC; ++q) acc[q] += valid ? x[j][q] * d_dx<BIN>(y[j][q]) : 0.f;
    }
  };

  walk_chunk<true, true>(
      a,
      [&](int) {
#pragma unroll
        for (int q = 0; q < VEC; ++q) acc[q] = 0.f;
      },
      [&](int32_t v, int32_t k, int, int cnt) {
        const float ys = (YM == kEdgeScalar && lane < cnt) ? __ldg(a.Y + k) : 0.f;
        int e0 = 0;
        for (; e0 + U * NG <= cnt; e0 += U * NG) step(True(), v, k, ys, e0, cnt);
        for (; e0 < cnt; e0 += U * NG) step(False(), v, k, ys, e0, cnt);
      },
      [&](int r, int slot) { store_sum<VEC>(a, acc, r, slot, f, 1, G, grp); });
}

// ---- dV of max / min ----
//
// Only n * F of the nnz * F (edge, feature) pairs are selected.  Comparing arg with the position of every
// edge, in the CSC's order, gathers a row of arg and a row of dO per edge (nnz * F * 8 bytes).  Instead
// arg_mask_kernel first walks the CSR and leaves `words` words per edge, bit j of word w set where the edge
// is feature f_lo + 32 w + j's extremum (arg is read once, nnz * words * 4 bytes are written); then
// general_dv_mask_kernel walks the CSC, reads the words of every edge, one random sector of 32 bytes, and of
// dO only the values that are selected.
// Bound by instruction issue and DRAM together (55 % and 65 % busy at 31 M edges, F = 100): about 20 instructions per
// edge with a selected feature, and a random sector per edge for its words beside the selected values.
// Both kernels, B200: 31 M edges F = 100 3.71 -> 1.59 ms; 16 M edges, columns up to 10^5, F = 128
// 4.28 -> 1.63 ms; 24 M edges F = 64 0.69 -> 0.41 ms; 5.7 M edges F = 602 5.73 -> 1.30 ms.

constexpr int kWindowWords = 1024;  // words of the mask a warp builds at a time

template <int WORDS>
__global__ void __launch_bounds__(kGenBlock) arg_mask_kernel(const GenArgs a) {
  constexpr int kEdges = kWindowWords / WORDS;
  __shared__ uint32_t windows[kGenWarps][kWindowWords];
  const int lane = threadIdx.x & 31;
  uint32_t* window = windows[threadIdx.x >> 5];
  const int chunk = blockIdx.x * kGenWarps + __shfl_sync(kAll, (int)(threadIdx.x >> 5), 0);
  if (chunk >= a.chunk_count) return;
  const int4 here = __ldg(reinterpret_cast<const int4*>(a.chunks) + chunk);
  const int4 next = __ldg(reinterpret_cast<const int4*>(a.chunks) + chunk + 1);
  const int nrows = here.z >= 0 ? 1 : next.x - here.x + (next.z >= 0 ? 1 : 0);
  int my_lo = 0, my_hi = 0;
  if (lane < nrows) {
    my_lo = max((int)__ldg(a.ptr + here.x + lane), here.y);
    my_hi = min((int)__ldg(a.ptr + here.x + lane + 1), next.y);
  }
  const int32_t* lane_arg = a.arg + (int64_t)here.x * a.F + a.f_lo + lane;
  const int width = min(32 * WORDS, a.F - a.f_lo) - lane;
  // the positions that row i selects, feature lane + 32 w in [w]; those of the next row are in flight
  auto load = [&](int i, int32_t (&k)[WORDS]) {
#pragma unroll
    for (int w = 0; w < WORDS; ++w)
      k[w] = i < nrows && 32 * w < width ? __ldg(lane_arg + (int64_t)i * a.F + 32 * w) : -1;
  };
  int32_t cur[WORDS], nxt[WORDS];
  load(0, cur);
  load(1, nxt);
  int i = 0;
  for (Position p0 = here.y; p0 < (Position)next.y; p0 += kEdges) {
    const Position p1 = min((Position)next.y, p0 + kEdges);
    for (int t = lane; t < (int)(p1 - p0) * WORDS; t += 32) window[t] = 0;
    __syncwarp();
    while (i < nrows) {
      const int lo = max(__shfl_sync(kAll, my_lo, i), (int)p0), end = __shfl_sync(kAll, my_hi, i);
      if (lo >= (int)p1) break;
      const int hi = min(end, (int)p1);
#pragma unroll
      for (int w = 0; w < WORDS; ++w)
        if (cur[w] >= lo && cur[w] < hi) atomicOr(&window[(cur[w] - (int)p0) * WORDS + w], 1u << lane);
      if (end > (int)p1) break;  // the rest of this row lies in the next window
      ++i;
#pragma unroll
      for (int w = 0; w < WORDS; ++w) cur[w] = nxt[w];
      load(i + 1, nxt);
    }
    __syncwarp();
    uint32_t* out = a.mask + (int64_t)p0 * WORDS;
    for (int t = lane; t < (int)(p1 - p0) * WORDS; t += 32) out[t] = window[t];
    __syncwarp();
  }
}

template <int WORDS>
__device__ __forceinline__ void load_mask(uint32_t (&m)[WORDS], const uint32_t* p) {
  if constexpr (WORDS == 1) {
    m[0] = __ldcs(p);
  } else if constexpr (WORDS == 2) {
    const uint2 v = __ldcs(reinterpret_cast<const uint2*>(p));
    m[0] = v.x; m[1] = v.y;
  } else {
#pragma unroll
    for (int q = 0; q < WORDS / 4; ++q) {
      const uint4 v = __ldcs(reinterpret_cast<const uint4*>(p) + q);
      m[4 * q] = v.x; m[4 * q + 1] = v.y; m[4 * q + 2] = v.z; m[4 * q + 3] = v.w;
    }
  }
}

// One edge's contribution to one feature: the selected value of dO times the derivative, or 0.
template <int BIN, int YM>
__device__ __forceinline__ float selected(const GenArgs& a, bool on, int64_t id, int64_t k, float ys, int f) {
  float x = load_if(on, a.X + id * a.ldx + f, 0.f);
  if (BIN == kMul || BIN == kDiv) {
    const float y = YM == kEdgeFull ? load_if(on, a.Y + k * a.F + f, 1.f) : ys;
    x = on ? x * d_dx<BIN>(y) : 0.f;
  }
  return x;
}

// More than 16 features: lane L holds the features f_lo + 32 w + L.  Edges without a selected feature are
// skipped, U of the others are in flight.
template <int BIN, int YM, int WORDS>
__global__ void __launch_bounds__(kGenBlock, WORDS > 4 ? 5 : 6) general_dv_mask_kernel(const GenArgs a) {
  constexpr int U = WORDS > 4 ? 2 : 4;
  const int lane = threadIdx.x & 31;
  const int f = a.f_lo + lane;
  float acc[WORDS];
  uint32_t ahead[WORDS];  // the words of the next batch's edges, a lane each
  walk_chunk<true, true>(
      a, [&](int32_t, int32_t k) { load_mask<WORDS>(ahead, a.mask + (int64_t)k * WORDS); },
      [&](int) {
#pragma unroll
        for (int w = 0; w < WORDS; ++w) acc[w] = 0.f;
      },
      [&](int32_t v, int32_t k, int, int cnt, int32_t, int32_t next_k) {
        uint32_t m[WORDS], any = 0;
#pragma unroll
        for (int w = 0; w < WORDS; ++w) {
          m[w] = lane < cnt ? ahead[w] : 0u;
          any |= m[w];
        }
        load_mask<WORDS>(ahead, a.mask + (int64_t)next_k * WORDS);
        float ys = 1.f;
        if (YM == kEdgeScalar) ys = load_if(any != 0, a.Y + k, 1.f);
        unsigned todo = __ballot_sync(kAll, any != 0);
        while (todo) {
          float x[U][WORDS];
#pragma unroll
          for (int t = 0; t < U; ++t) {
            const int e = (__ffs(todo) - 1) & 31;
            const uint32_t some = todo ? 0xffffffffu : 0u;
            todo &= todo - 1u;
            const int32_t id = __shfl_sync(kAll, v, e);
            const int32_t pos = YM == kEdgeFull ? __shfl_sync(kAll, k, e) : 0;
            const float y = YM == kEdgeScalar ? __shfl_sync(kAll, ys, e) : 1.f;
#pragma unroll
            for (int w = 0; w < WORDS; ++w) {
              const uint32_t word = __shfl_sync(kAll, m[w], e) & some;
              x[t][w] = selected<BIN, YM>(a, (word >> lane) & 1u, id, pos, y, f + 32 * w);
            }
          }
#pragma unroll
          for (int t = 0; t < U; ++t)
#pragma unroll
            for (int w = 0; w < WORDS; ++w) acc[w] += x[t][w];
        }
      },
      [&](int r, int slot) { store_sum<WORDS>(a, acc, r, slot, f, 32, 32, 0); });
}

// Up to 16 features: groups of G lanes take an edge each.
template <int BIN, int YM>
__global__ void __launch_bounds__(kGenBlock, 6) general_dv_mask_narrow_kernel(const GenArgs a) {
  constexpr int U = 2;
  const int lane = threadIdx.x & 31;
  const int G = 1 << a.log_g, NG = 32 >> a.log_g;
  const int grp = lane >> a.log_g, c = lane & (G - 1);
  float acc[1];
  uint32_t ahead[1];
  walk_chunk<true, true>(
      a, [&](int32_t, int32_t k) { load_mask<1>(ahead, a.mask + k); }, [&](int) { acc[0] = 0.f; },
      [&](int32_t v, int32_t k, int, int cnt, int32_t, int32_t next_k) {
        const uint32_t m = lane < cnt ? ahead[0] : 0u;
        load_mask<1>(ahead, a.mask + next_k);
        const float ys = YM == kEdgeScalar ? load_if(m != 0, a.Y + k, 1.f) : 1.f;
        for (int e0 = 0; e0 < cnt; e0 += U * NG) {
          float x[U];
#pragma unroll
          for (int t = 0; t < U; ++t) {
            const int e = e0 + t * NG + grp;
            uint32_t word = __shfl_sync(kAll, m, e & 31);
            if (e >= 32) word = 0;
            x[t] = selected<BIN, YM>(a, (word >> c) & 1u, __shfl_sync(kAll, v, e & 31), __shfl_sync(kAll, k, e & 31),
                                     YM == kEdgeScalar ? __shfl_sync(kAll, ys, e & 31) : 1.f, c);
          }
#pragma unroll
          for (int t = 0; t < U; ++t) acc[0] += x[t];
        }
      },
      [&](int r, int slot) { store_sum<1>(a, acc, r, slot, c, 1, G, grp); });
}

// The same without a mask (see mask_pays, or no memory for it): arg itself is compared, four features per lane.
template <int BIN, int YM, int VEC>
__global__ void __launch_bounds__(kGenBlock, 4) general_dv_extremum_kernel(const GenArgs a) {
  constexpr int U = 4;
  const int lane = threadIdx.x & 31;
  const int G = 1 << a.log_g, NG = 32 >> a.log_g;
  const int grp = lane >> a.log_g, c = lane & (G - 1);
  const int f = (blockIdx.y + a.first_slice) * (G * 4) + c * 4;
  const int room = f < a.F ? min(4, a.F - f) : 0;
  const int fl = room ? f : 0;
  float acc[4];
  walk_chunk<true, true>(
      a,
      [&](int) {
#pragma unroll
        for (int q = 0; q < 4; ++q) acc[q] = 0.f;
      },
      [&](int32_t v, int32_t k, int, int cnt) {
        for (int e0 = 0; e0 < cnt; e0 += U * NG) {
          int32_t id[U], pos[U], sel[U][4];
          float x[U][4];
#pragma unroll
          for (int j = 0; j < U; ++j) {
            const int e = e0 + j * NG + grp;
            id[j] = __shfl_sync(kAll, v, e & 31);
            pos[j] = __shfl_sync(kAll, k, e & 31);
            const int32_t* row = a.arg + (int64_t)id[j] * a.F + fl;
            if constexpr (VEC == 4) {
              load_vec<4>(sel[j], row);
            } else {
#pragma unroll
              for (int q = 0; q < 4; ++q) sel[j][q] = __ldg(row + (q < room ? q : 0));
            }
#pragma unroll
            for (int q = 0; q < 4; ++q)
              if (e >= cnt || q >= room) sel[j][q] = -1;
          }
#pragma unroll
          for (int j = 0; j < U; ++j)
#pragma unroll
            for (int q = 0; q < 4; ++q) {
              const float ys =
                  YM == kEdgeScalar ? load_if(sel[j][q] == pos[j], a.Y + pos[j], 1.f) : 1.f;
              x[j][q] = selected<BIN, YM>(a, sel[j][q] == pos[j], id[j], pos[j], ys, fl + q);
            }
#pragma unroll
          for (int j = 0; j < U; ++j)
#pragma unroll
            for (int q = 0; q < 4; ++q) acc[q] += x[j][q];
        }
      },
      [&](int r, int slot) { store_sum<4>(a, acc, r, slot, f, 1, G, grp); });
}

// dE with full edge features: one value per (edge, feature).  The written rows, nnz * F floats in CSR
// order, are the traffic: streaming stores leave L2 to the gathered rows.
template <int BIN, int RED, int VEC, int U>
__global__ void __launch_bounds__(kGenBlock) general_de_full_kernel(const GenArgs a) {
  constexpr bool kNeedsX = BIN == kMul || BIN == kDiv;
  const int lane = threadIdx.x & 31;
  const int G = 1 << a.log_g, NG = 32 >> a.log_g;
  const int grp = lane >> a.log_g, c = lane & (G - 1);
  const int f = blockIdx.y * (G * VEC) + c * VEC;
  const bool on = f < a.F;
  const int fl = on ? f : 0;
  float g[VEC];
  int32_t sel[VEC];
  walk_chunk<kNeedsX, false>(
      a,
      [&](int r) {
        load_vec<VEC>(g, a.X + (int64_t)r * a.F + fl);
        if (RED != kSum) load_vec<VEC>(sel, a.arg + (int64_t)r * a.F + fl);
      },
      [&](int32_t u, int32_t, int b, int cnt) {
        for (int e0 = 0; e0 < cnt; e0 += U * NG) {
          float x[U][VEC], y[U][VEC];
#pragma unroll
          for (int j = 0; j < U; ++j) {
            const int e = e0 + j * NG + grp;
#pragma unroll
            for (int q = 0; q < VEC; ++q) {
              x[j][q] = 0.f;
              y[j][q] = BIN == kDiv ? 1.f : 0.f;  // absent edges: a division by zero takes a slow path
            }
            if (kNeedsX) {
              const int32_t id = __shfl_sync(kAll, u, e & 31);
              if (e < cnt) load_vec<VEC>(x[j], a.V + (int64_t)id * a.F + fl);
            }
            if (BIN == kDiv && e < cnt) stream_vec<VEC>(y[j], a.Y + (int64_t)(b + e) * a.F + fl);
          }
#pragma unroll
          for (int j = 0; j < U; ++j) {
            const int e = e0 + j * NG + grp;
            float t[VEC];
#pragma unroll
            for (int q = 0; q < VEC; ++q) {
              t[q] = g[q] * d_dy<BIN>(x[j][q], y[j][q]);
              if (RED != kSum && sel[q] != b + e) t[q] = 0.f;
            }
            if (!on || e >= cnt) continue;
            float* o = a.out + (int64_t)(b + e) * a.F + f;
            if constexpr (VEC == 4)
              __stcs(reinterpret_cast<float4*>(o), make_float4(t[0], t[1], t[2], t[3]));
            else
              __stcs(o, t[0]);
          }
        }
      },
      [](int, int) {});
}

// dE with one column (the broadcast scalar): the feature sum of the above, one dot product per edge reduced
// inside the lane group.  (mul / sum runs on the edge-weight gradient, dg_edge_grad.cu.)
template <int BIN, int RED>
__global__ void __launch_bounds__(kGenBlock) general_de_scalar_kernel(const GenArgs a) {
  constexpr bool kNeedsX = BIN == kMul || BIN == kDiv;
  const int lane = threadIdx.x & 31;
  const int G = 1 << a.log_g, NG = 32 >> a.log_g;
  const int grp = lane >> a.log_g, c = lane & (G - 1);
  const int F = a.F;
  int64_t row = 0;
  walk_chunk<kNeedsX, false>(
      a, [&](int r) { row = r; },
      [&](int32_t u, int32_t, int b, int cnt) {
        for (int e0 = 0; e0 < cnt; e0 += NG) {
          const int e = e0 + grp;
          const int32_t id = __shfl_sync(kAll, u, e & 31);
          float dot = 0.f;
          if (e < cnt) {
            const float y = BIN == kDiv ? __ldg(a.Y + b + e) : 0.f;
            for (int j = c; j < F; j += G) {
              float t = __ldg(a.X + row * F + j) * d_dy<BIN>(kNeedsX ? __ldg(a.V + (int64_t)id * F + j) : 0.f, y);
              if (RED != kSum && __ldg(a.arg + row * F + j) != b + e) t = 0.f;
              dot += t;
            }
          }
          for (int off = 1; off < G; off <<= 1) dot += __shfl_xor_sync(kAll, dot, off);
          if (e < cnt && c == 0) a.out[b + e] = dot;
        }
      },
      [](int, int) {});
}

dg_status_t launched() {
  DG_CUDA(cudaGetLastError());
  count_launches(1);
  return DG_OK;
}

unsigned chunk_blocks(const GenArgs& a) { return (unsigned)((a.chunk_count + kGenWarps - 1) / kGenWarps); }

template <int BIN, int YM, int VEC>
dg_status_t launch_dv_sum(const GenArgs& a, cudaStream_t s) {
  const dim3 grid = general_grid(a, VEC);
  if (a.log_g >= 3) general_dv_sum_kernel<BIN, YM, VEC, 4><<<grid, kGenBlock, 0, s>>>(a);
  else if (a.log_g >= 1) general_dv_sum_kernel<BIN, YM, VEC, 2><<<grid, kGenBlock, 0, s>>>(a);
  else general_dv_sum_kernel<BIN, YM, VEC, 1><<<grid, kGenBlock, 0, s>>>(a);  // a batch is one step
  return launched();
}

template <int BIN, int YM>
dg_status_t launch_dv_extremum(const GenArgs& a, cudaStream_t s) {
  if (a.mask) {
    const unsigned grid = chunk_blocks(a);
    if (a.F <= 16) general_dv_mask_narrow_kernel<BIN, YM><<<grid, kGenBlock, 0, s>>>(a);
    else if (a.words == 1) general_dv_mask_kernel<BIN, YM, 1><<<grid, kGenBlock, 0, s>>>(a);
    else if (a.words == 2) general_dv_mask_kernel<BIN, YM, 2><<<grid, kGenBlock, 0, s>>>(a);
    else if (a.words == 4) general_dv_mask_kernel<BIN, YM, 4><<<grid, kGenBlock, 0, s>>>(a);
    else general_dv_mask_kernel<BIN, YM, 8><<<grid, kGenBlock, 0, s>>>(a);
  } else {
    const dim3 grid = general_grid(a, 4);
    if (a.vec == 4) general_dv_extremum_kernel<BIN, YM, 4><<<grid, kGenBlock, 0, s>>>(a);
    else general_dv_extremum_kernel<BIN, YM, 1><<<grid, kGenBlock, 0, s>>>(a);
  }
  return launched();
}

template <int BIN>
dg_status_t dv_by_reducer(const GenArgs& a, int red, cudaStream_t s) {
  constexpr bool kNeedsY = BIN == kMul || BIN == kDiv;
  if (red == kSum) {
    if constexpr (kNeedsY) {
      if (a.cols != 1) {
        if (a.vec == 4) return launch_dv_sum<BIN, kEdgeFull, 4>(a, s);
        if (a.vec == 2) return launch_dv_sum<BIN, kEdgeFull, 2>(a, s);
        return launch_dv_sum<BIN, kEdgeFull, 1>(a, s);
      }
      if (a.vec == 4) return launch_dv_sum<BIN, kEdgeScalar, 4>(a, s);
      if (a.vec == 2) return launch_dv_sum<BIN, kEdgeScalar, 2>(a, s);
      return launch_dv_sum<BIN, kEdgeScalar, 1>(a, s);
    } else {
      return DG_ERR_UNSUPPORTED;  // dg_ap_bwd hands these pairs to aggregate_sum
    }
  }
  // The reducer plays no part beyond its arg: max and min share the kernels.  So do copylhs, add and sub,
  // whose derivative is 1.
  if constexpr (kNeedsY) {
    if (a.cols != 1) return launch_dv_extremum<BIN, kEdgeFull>(a, s);
    return launch_dv_extremum<BIN, kEdgeScalar>(a, s);
  } else {
    return launch_dv_extremum<kCopyLhs, kNoEdge>(a, s);
  }
}

// A batch has 32 edges, which narrow groups cover in fewer steps: what is left over would only divide (gradients of
// div / sum with full edge features, F = 4: 7.9 M edges 452 us with four steps and zero divisors, 199 so).
template <int BIN, int RED, int VEC>
void launch_de_full(const GenArgs& a, cudaStream_t s) {
  const dim3 grid = general_grid(a, VEC);
  if (a.log_g >= 2) general_de_full_kernel<BIN, RED, VEC, 4><<<grid, kGenBlock, 0, s>>>(a);
  else if (a.log_g == 1) general_de_full_kernel<BIN, RED, VEC, 2><<<grid, kGenBlock, 0, s>>>(a);
  else general_de_full_kernel<BIN, RED, VEC, 1><<<grid, kGenBlock, 0, s>>>(a);
}

template <int BIN, int RED>
dg_status_t launch_de(const GenArgs& a, cudaStream_t s) {
  if (a.cols == 1) general_de_scalar_kernel<BIN, RED><<<chunk_blocks(a), kGenBlock, 0, s>>>(a);
  else if (a.vec == 4) launch_de_full<BIN, RED, 4>(a, s);
  else launch_de_full<BIN, RED, 1>(a, s);
  return launched();
}

template <int BIN>
dg_status_t de_by_reducer(const GenArgs& a, int red, cudaStream_t s) {
  return red == kSum ? launch_de<BIN, kSum>(a, s) : launch_de<BIN, kMax>(a, s);  // max and min share
}

}  // namespace

dg_status_t launch_general_dv(const GenArgs& a, int bin, int red, cudaStream_t s) {
  switch (bin) {
    case kMul: return dv_by_reducer<kMul>(a, red, s);
    case kDiv: return dv_by_reducer<kDiv>(a, red, s);
    default: return dv_by_reducer<kCopyLhs>(a, red, s);
  }
}

dg_status_t launch_general_de(const GenArgs& a, int bin, int red, cudaStream_t s) {
  switch (bin) {
    case kSub: return de_by_reducer<kSub>(a, red, s);
    case kMul: return de_by_reducer<kMul>(a, red, s);
    case kDiv: return de_by_reducer<kDiv>(a, red, s);
    default: return de_by_reducer<kCopyRhs>(a, red, s);  // add and copyrhs: the derivative is 1
  }
}

dg_status_t launch_arg_mask(const GenArgs& a, cudaStream_t s) {
  const unsigned grid = chunk_blocks(a);
  if (a.words == 1) arg_mask_kernel<1><<<grid, kGenBlock, 0, s>>>(a);
  else if (a.words == 2) arg_mask_kernel<2><<<grid, kGenBlock, 0, s>>>(a);
  else if (a.words == 4) arg_mask_kernel<4><<<grid, kGenBlock, 0, s>>>(a);
  else arg_mask_kernel<8><<<grid, kGenBlock, 0, s>>>(a);
  return launched();
}

}  // namespace dg
