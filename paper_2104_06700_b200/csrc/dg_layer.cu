// Elementwise passes around the GEMM of a GraphSAGE layer,  out = act(D Z + b)  with D a diagonal matrix, and
// their gradients.  D (Z W) = (D Z) W, so the division by the in-degree needs no pass over n x F of its own in
// either direction: forward it rides with bias and ReLU, backward with the mask and the sums of the bias.
//
// Both kernels are streams.  245 k rows of 256: forward 0.5 GB, backward 0.75 GB.
#include "dg_internal.cuh"

namespace dg {
namespace {

constexpr int kStreamBlock = 256;
// Rows in flight per thread: four 16-byte loads of each operand cover the latency with 8 blocks per SM.
constexpr int kStreamRows = 4;
constexpr int kStreamBlocksPerSm = 8;

template <int VEC>
struct Pack {
  float v[VEC];
};
template <int VEC>
__device__ __forceinline__ Pack<VEC> load_pack(const float* p) {
  Pack<VEC> r;
  if constexpr (VEC == 4) {
    const float4 q = *reinterpret_cast<const float4*>(p);
    r.v[0] = q.x, r.v[1] = q.y, r.v[2] = q.z, r.v[3] = q.w;
  } else {
    r.v[0] = *p;
  }
  return r;
}
template <int VEC>
__device__ __forceinline__ void store_pack(float* p, const Pack<VEC>& r) {
  if constexpr (VEC == 4) {
    *reinterpret_cast<float4*>(p) = make_float4(r.v[0], r.v[1], r.v[2], r.v[3]);
  } else {
    *p = r.v[0];
  }
}

// A thread owns VEC columns (blockIdx.y: the tile of blockDim.x vectors) and every blockDim.y * gridDim.x-th
// row, so that the bias, and backward the sum of its gradient, stay in registers.
template <int VEC>
__global__ void __launch_bounds__(kStreamBlock)
    layer_fwd_kernel(float* Y, const float* scale, const float* bias, int64_t n, int32_t F, bool relu) {
  const int32_t f = (blockIdx.y * blockDim.x + threadIdx.x) * VEC;
  if (f >= F) return;
  const Pack<VEC> b = load_pack<VEC>(bias + f);
  const int64_t step = (int64_t)gridDim.x * blockDim.y;
  for (int64_t r0 = (int64_t)blockIdx.x * blockDim.y + threadIdx.y; r0 < n; r0 += step * kStreamRows) {
    Pack<VEC> y[kStreamRows];
    float s[kStreamRows];
#pragma unroll
    for (int u = 0; u < kStreamRows; ++u) {
      const int64_t r = r0 + u * step;
      if (r < n) {
        y[u] = load_pack<VEC>(Y + r * F + f);
        s[u] = scale[r];
      }
    }
#pragma unroll
    for (int u = 0; u < kStreamRows; ++u) {
      const int64_t r = r0 + u * step;
      if (r >= n) break;
#pragma unroll
      for (int c = 0; c < VEC; ++c) {
        const float v = y[u].v[c] * s[u] + b.v[c];
        y[u].v[c] = relu && v <= 0.f ? 0.f : v;  // NaN stays NaN
      }
      store_pack<VEC>(Y + r * F + f, y[u]);
    }
  }
}

// G = D (dOut where out > 0), and into partial[blockIdx.x] (unless null) the column sums of the masked dOut over the
// block's rows.  `out` null: no mask.
template <int VEC>
__global__ void __launch_bounds__(kStreamBlock)
    layer_bwd_kernel(const float* dOut, const float* out, const float* scale, int64_t n, int32_t F, float* G,
                     float* partial) {
  __shared__ float sums[kStreamBlock * VEC];
  const int32_t f = (blockIdx.y * blockDim.x + threadIdx.x) * VEC;
  float total[VEC] = {};
  const int64_t step = (int64_t)gridDim.x * blockDim.y;
  if (f < F) {
    for (int64_t r0 = (int64_t)blockIdx.x * blockDim.y + threadIdx.y; r0 < n; r0 += step * kStreamRows) {
      Pack<VEC> d[kStreamRows], o[kStreamRows];
      float s[kStreamRows];
#pragma unroll
      for (int u = 0; u < kStreamRows; ++u) {
        const int64_t r = r0 + u * step;
        if (r < n) {
          d[u] = load_pack<VEC>(dOut + r * F + f);
          if (out) o[u] = load_pack<VEC>(out + r * F + f);
          s[u] = scale[r];
        }
      }
#pragma unroll
      for (int u = 0; u < kStreamRows; ++u) {
        const int64_t r = r0 + u * step;
        if (r >= n) break;
#pragma unroll
        for (int c = 0; c < VEC; ++c) {
          const float v = out && o[u].v[c] <= 0.f ? 0.f : d[u].v[c];
          total[c] += v;
          d[u].v[c] = v * s[u];
        }
        store_pack<VEC>(G + r * F + f, d[u]);
      }
    }
  }
  if (!partial) return;
#pragma unroll
  for (int c = 0; c < VEC; ++c) sums[(threadIdx.y * VEC + c) * blockDim.x + threadIdx.x] = total[c];
  __syncthreads();
  if (threadIdx.y == 0 && f < F) {
#pragma unroll
    for (int c = 0; c < VEC; ++c) {
      float t = 0.f;
      for (int y = 0; y < (int)blockDim.y; ++y) t += sums[(y * VEC + c) * blockDim.x + threadIdx.x];
      partial[(int64_t)blockIdx.x * F + f + c] = t;
    }
  }
}

// dbias[f] = the sum over the blocks, always in the same order: 32 columns x 32 threads per block.
__global__ void __launch_bounds__(1024) layer_bias_kernel(const float* partial, int32_t blocks, int32_t F,
                                                          float* dbias) {
  __shared__ float sums[32][33];
  const int32_t f = blockIdx.x * 32 + threadIdx.x;
  float t = 0.f;
  if (f < F)
    for (int32_t b = threadIdx.y; b < blocks; b += 32) t += partial[(int64_t)b * F + f];
  sums[threadIdx.y][threadIdx.x] = t;
  __syncthreads();
  t = sums[threadIdx.x][threadIdx.y];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
  const int32_t column = blockIdx.x * 32 + threadIdx.y;
  if (threadIdx.x == 0 && column < F) dbias[column] = t;
}

// dbias from dOut itself, where there is no memory for the blocks' sums: 32 columns x 32 threads per block again, the
// sum of every 64 rows of a thread added to its total.
__global__ void __launch_bounds__(1024) layer_bias_direct_kernel(const float* dOut, const float* out, int64_t n,
                                                                 int32_t F, float* dbias) {
  __shared__ float sums[32][33];
  const int32_t f = blockIdx.x * 32 + threadIdx.x;
  float t = 0.f;
  if (f < F) {
    for (int64_t r0 = threadIdx.y; r0 < n; r0 += 64 * 32) {
      float part = 0.f;
      for (int64_t r = r0; r < n && r < r0 + 64 * 32; r += 32) {
        const float d = dOut[r * F + f];
        part += out && out[r * F + f] <= 0.f ? 0.f : d;
      }
      t += part;
    }
  }
  sums[threadIdx.y][threadIdx.x] = t;
  __syncthreads();
  t = sums[threadIdx.x][threadIdx.y];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
  const int32_t column = blockIdx.x * 32 + threadIdx.y;
  if (threadIdx.x == 0 && column < F) dbias[column] = t;
}

// Threads along the columns: the power of two that covers a row, at most a block; the rest along the rows.
void stream_shape(const Graph* g, int32_t F, int vec, dim3* grid, dim3* block) {
  const int32_t vectors = F / vec;
  int x = 1;
  while (x < vectors && x < kStreamBlock) x *= 2;
  const int y = kStreamBlock / x;
  const int64_t tiles = (vectors + x - 1) / x;
  int64_t blocks = (g->n + (int64_t)y * kStreamRows - 1) / ((int64_t)y * kStreamRows);
  const int64_t most = (int64_t)g->sm_count * kStreamBlocksPerSm / tiles;
  if (blocks > most) blocks = most;
  if (blocks < 1) blocks = 1;
  *block = dim3((unsigned)x, (unsigned)y);
  *grid = dim3((unsigned)blocks, (unsigned)tiles);
}

bool aligned16(const void* p) { return reinterpret_cast<uintptr_t>(p) % 16 == 0; }

}  // namespace

dg_status_t layer_fwd(const Graph* g, float* Y, int32_t F, const float* scale, const float* bias, bool relu,
                      cudaStream_t s) {
  const bool wide = F % 4 == 0 && aligned16(Y) && aligned16(bias);
  dim3 grid, block;
  stream_shape(g, F, wide ? 4 : 1, &grid, &block);
  if (wide)
    layer_fwd_kernel<4><<<grid, block, 0, s>>>(Y, scale, bias, g->n, F, relu);
  else
    layer_fwd_kernel<1><<<grid, block, 0, s>>>(Y, scale, bias, g->n, F, relu);
  DG_CUDA(cudaGetLastError());
  count_launches(1);
  return DG_OK;
}

dg_status_t layer_bwd(const Graph* g, const float* dOut, const float* out, int32_t F, const float* scale,
                      float* G, float* dbias, cudaStream_t s) {
  const bool wide = F % 4 == 0 && aligned16(dOut) && aligned16(G) && (!out || aligned16(out));
  dim3 grid, block;
  stream_shape(g, F, wide ? 4 : 1, &grid, &block);
  void* partial = nullptr;
  const unsigned columns = (unsigned)((F + 31) / 32);
  if (scratch_alloc(g, (size_t)grid.x * (size_t)F * sizeof(float), s, &partial) != cudaSuccess)
    // first: G may take the place of dOut
    layer_bias_direct_kernel<<<columns, dim3(32, 32), 0, s>>>(dOut, out, g->n, F, dbias);
  float* sums = static_cast<float*>(partial);
  if (wide)
    layer_bwd_kernel<4><<<grid, block, 0, s>>>(dOut, out, scale, g->n, F, G, sums);
  else
    layer_bwd_kernel<1><<<grid, block, 0, s>>>(dOut, out, scale, g->n, F, G, sums);
  if (sums) layer_bias_kernel<<<columns, dim3(32, 32), 0, s>>>(sums, (int32_t)grid.x, F, dbias);
  const cudaError_t e = cudaGetLastError();
  pool_free(partial, s);
  DG_CUDA(e);
  count_launches(2);
  return DG_OK;
}

}  // namespace dg
