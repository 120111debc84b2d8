// Softmax cross-entropy over some rows of an n x C matrix (the training vertices of an epoch) and its gradient
// with respect to the whole matrix.
//
// 163 k rows of 47 classes are 31 MB in L2: what bounds both kernels is the chain index -> row -> reduction,
// so a warp reads the indices and labels of 16 rows at once and has the loads of four rows in flight.
#include "dg_internal.cuh"

namespace dg {
namespace {

constexpr int kLossBlock = 256;
constexpr int kRowsPerWarp = 16;
constexpr int kRowsPerBlock = kLossBlock / 32 * kRowsPerWarp;
constexpr int64_t kIgnored = -100;  // label of a row that does not count
constexpr unsigned kAll = 0xffffffffu;

// row < 0: the row does not count; `bad`: its index or label is out of range.
struct Target {
  int64_t row;
  int32_t label;
  bool bad;
};
__device__ __forceinline__ Target target_of(const int64_t* index, const int64_t* labels, int64_t t,
                                            int64_t count, int64_t n, int32_t C) {
  Target r{-1, 0, false};
  if (t >= count) return r;
  int64_t v = index[t];
  if (v < 0) v += n;
  if (v < 0 || v >= n) {
    r.bad = true;
    return r;
  }
  const int64_t y = labels[v];
  if (y == kIgnored) return r;
  if (y < 0 || y >= C) {
    r.bad = true;
    return r;
  }
  r.row = v;
  r.label = (int32_t)y;
  return r;
}

__device__ __forceinline__ float warp_max(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const float w = __shfl_xor_sync(kAll, v, o);
    v = v > w || v != v ? v : w;  // NaN stays
  }
  return v;
}
template <typename T>
__device__ __forceinline__ T warp_sum(T v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kAll, v, o);
  return v;
}

// K registers per lane hold a row of up to 32 K classes; K = 0 reads it twice.  stats[t] = (max, log of the sum
// of exp(x - max)).  Each of `shares` (128 rows) leaves partial[share] = (sum of the losses, rows that count; NaN after
// a bad index or label).  Without memory for them (partial null) one block takes all shares and writes the result.
template <int K>
__global__ void __launch_bounds__(kLossBlock)
    loss_fwd_kernel(const float* __restrict__ logits, int64_t n, int32_t C, const int64_t* __restrict__ index,
                    int64_t count, const int64_t* __restrict__ labels, float2* __restrict__ stats,
                    double2* __restrict__ partial, int64_t shares, float* __restrict__ result) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x / 32;
  __shared__ double losses[kLossBlock / 32];
  __shared__ int counts[kLossBlock / 32];
  double2 all = make_double2(0.0, 0.0);
  for (int64_t share = blockIdx.x; share < shares; share += gridDim.x) {
    const int64_t t0 = share * kRowsPerBlock + warp * kRowsPerWarp;
    const Target mine = target_of(index, labels, lane < kRowsPerWarp ? t0 + lane : count, count, n, C);
    const int64_t my_row = mine.row < 0 ? 0 : mine.row;
    float my_max = 0.f, my_log = 0.f, my_target = 0.f;
#pragma unroll 4
    for (int j = 0; j < kRowsPerWarp; ++j) {
      const float* x = logits + __shfl_sync(kAll, my_row, j) * C;
      float m = -INFINITY, s = 0.f;
      if constexpr (K > 0) {
        float v[K > 0 ? K : 1];
#pragma unroll
        for (int k = 0; k < K; ++k) {
          const int c = lane + 32 * k;
          v[k] = c < C ? x[c] : -INFINITY;
          m = m > v[k] || m != m ? m : v[k];
        }
        m = warp_max(m);
#pragma unroll
        for (int k = 0; k < K; ++k) s += lane + 32 * k < C ? expf(v[k] - m) : 0.f;
      } else {
        for (int c = lane; c < C; c += 32) m = m > x[c] || m != m ? m : x[c];
        m = warp_max(m);
        for (int c = lane; c < C; c += 32) s += expf(x[c] - m);
      }
      s = warp_sum(s);
      if (lane == j) {
        my_max = m;
        my_log = logf(s);
      }
    }
    if (lane < kRowsPerWarp && t0 + lane < count) {
      my_target = logits[my_row * C + mine.label];
      stats[t0 + lane] = make_float2(my_max, my_log);
    }
    double loss = mine.row >= 0 ? (double)((my_max - my_target) + my_log) : 0.0;
    if (mine.bad) loss = NAN;
    loss = warp_sum(loss);
    const int rows = __popc(__ballot_sync(kAll, mine.row >= 0));
    if (lane == 0) {
      losses[warp] = loss;
      counts[warp] = rows;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
      double l = 0.0;
      int r = 0;
      for (int i = 0; i < kLossBlock / 32; ++i) {
        l += losses[i];
        r += counts[i];
      }
      if (partial) partial[share] = make_double2(l, (double)r);
      all.x += l;
      all.y += (double)r;
    }
    __syncthreads();
  }
  if (!partial && threadIdx.x == 0) {
    result[0] = (float)(all.x / all.y);
    result[1] = (float)(1.0 / all.y);
  }
}

// result = (mean loss, 1 / rows that count)
__global__ void __launch_bounds__(1024) loss_mean_kernel(const double2* __restrict__ partial, int64_t blocks,
                                                         float* __restrict__ result) {
  double loss = 0.0, rows = 0.0;
  for (int64_t b = threadIdx.x; b < blocks; b += 1024) {
    const double2 p = partial[b];
    loss += p.x;
    rows += p.y;
  }
  __shared__ double2 sums[32];
  loss = warp_sum(loss);
  rows = warp_sum(rows);
  if (threadIdx.x % 32 == 0) sums[threadIdx.x / 32] = make_double2(loss, rows);
  __syncthreads();
  if (threadIdx.x < 32) {
    const double2 p = sums[threadIdx.x];
    loss = warp_sum(p.x);
    rows = warp_sum(p.y);
    if (threadIdx.x == 0) {
      result[0] = (float)(loss / rows);  // no rows: NaN
      result[1] = (float)(1.0 / rows);
    }
  }
}

// d += (softmax - one-hot) * grad / rows on the rows of `index`.  A row named twice gets its gradient twice: the
// atomic additions of equal terms give the same sum in any order.
__global__ void __launch_bounds__(kLossBlock)
    loss_bwd_kernel(const float* __restrict__ logits, int64_t n, int32_t C, const int64_t* __restrict__ index,
                    int64_t count, const int64_t* __restrict__ labels, const float2* __restrict__ stats,
                    const float* __restrict__ result, const float* __restrict__ grad, float* __restrict__ d) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x / 32;
  const int64_t t0 = (int64_t)blockIdx.x * kRowsPerBlock + warp * kRowsPerWarp;
  const Target mine = target_of(index, labels, lane < kRowsPerWarp ? t0 + lane : count, count, n, C);
  const float2 my_stats = mine.row >= 0 ? stats[t0 + lane] : make_float2(0.f, 0.f);
  const float scale = *grad * result[1];
#pragma unroll 4
  for (int j = 0; j < kRowsPerWarp; ++j) {
    const int64_t row = __shfl_sync(kAll, mine.row, j);
    const int32_t label = __shfl_sync(kAll, mine.label, j);
    const float m = __shfl_sync(kAll, my_stats.x, j), log_sum = __shfl_sync(kAll, my_stats.y, j);
    if (row < 0) continue;
    for (int32_t c = lane; c < C; c += 32) {
      const float p = expf((logits[row * C + c] - m) - log_sum);
      atomicAdd(d + row * C + c, (c == label ? p - 1.f : p) * scale);
    }
  }
}

unsigned loss_blocks(int64_t count) { return (unsigned)((count + kRowsPerBlock - 1) / kRowsPerBlock); }

}  // namespace

dg_status_t loss_fwd(const Graph* g, const float* logits, int32_t C, const int64_t* index, int64_t count,
                     const int64_t* labels, float* stats, float* result, cudaStream_t s) {
  const unsigned blocks = loss_blocks(count);
  void* memory = nullptr;
  const bool missing = blocks && scratch_alloc(g, blocks * sizeof(double2), s, &memory) != cudaSuccess;
  double2* partial = static_cast<double2*>(memory);
  float2* st = reinterpret_cast<float2*>(stats);
  if (blocks) {
    auto kernel = C <= 32 ? loss_fwd_kernel<1> : C <= 64 ? loss_fwd_kernel<2> : C <= 128 ? loss_fwd_kernel<4>
                                                                                        : loss_fwd_kernel<0>;
    kernel<<<missing ? 1 : blocks, kLossBlock, 0, s>>>(logits, g->n, C, index, count, labels, st, partial, blocks, result);
  }
  if (!missing) loss_mean_kernel<<<1, 1024, 0, s>>>(partial, blocks, result);
  const cudaError_t e = cudaGetLastError();
  pool_free(memory, s);
  DG_CUDA(e);
  count_launches(blocks && !missing ? 2 : 1);
  return DG_OK;
}

dg_status_t loss_bwd(const Graph* g, const float* logits, int32_t C, const int64_t* index, int64_t count,
                     const int64_t* labels, const float* stats, const float* result, const float* grad,
                     float* d, cudaStream_t s) {
  if (g->n == 0) return DG_OK;
  DG_CUDA(cudaMemsetAsync(d, 0, (size_t)g->n * (size_t)C * sizeof(float), s));
  const unsigned blocks = loss_blocks(count);
  if (blocks == 0) return DG_OK;
  loss_bwd_kernel<<<blocks, kLossBlock, 0, s>>>(logits, g->n, C, index, count, labels,
                                                reinterpret_cast<const float2*>(stats), result, grad, d);
  DG_CUDA(cudaGetLastError());
  count_launches(1);
  return DG_OK;
}

}  // namespace dg
