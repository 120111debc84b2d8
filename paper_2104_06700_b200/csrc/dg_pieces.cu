// The later pieces of cut rows without scratch memory.  A call normally leaves their results in slots of a scratch
// array and joins them; when the library's pool cannot give that array (or the handle's "scratch_mb" forbids it), the
// main kernels leave these pieces out and this kernel adds them to what the first piece of a row stored.
//
// A warp takes a row and 32 features, piece after piece: slower than the slots by a factor of several on a hub, but it
// runs only where the call would otherwise fail.  A piece is summed before it is added (pieces of at most two chunks),
// so a hub is not one long chain of fp32 additions.
#include "dg_general.cuh"

namespace dg {
namespace {

__device__ float gathered(const PieceArgs& a, int32_t id, int f) {
  const int64_t i = (int64_t)id * a.ldx + f;
  if (a.bf16) return __uint_as_float((uint32_t)__ldg(static_cast<const uint16_t*>(a.X) + i) << 16);
  return __ldg(static_cast<const float*>(a.X) + i);
}

__device__ float message_of(int bin, float x, float y) {
  switch (bin) {
    case kCopyRhs: return message<kCopyRhs>(x, y);
    case kAdd: return message<kAdd>(x, y);
    case kSub: return message<kSub>(x, y);
    case kMul: return message<kMul>(x, y);
    case kDiv: return message<kDiv>(x, y);
    default: return x;
  }
}

constexpr int kGroup = 32;  // pieces that are added before they go to the total

__global__ void __launch_bounds__(32) pieces_kernel(const PieceArgs a) {
  const int f = blockIdx.y * 32 + threadIdx.x;
  if (f >= a.F) return;
  const int cut_rows = min(__ldg(a.totals + 1), a.max_cuts);
  for (int i = blockIdx.x; i < cut_rows; i += gridDim.x) {
    const CutRow cut = a.cuts[i];
    const int64_t o = (int64_t)cut.row * a.F + f;
    float total = 0.f, group = 0.f;
    float best = a.red == kSum ? 0.f : a.out[o];
    int32_t at = a.red != kSum && a.arg_out ? a.arg_out[o] : 0;
    for (int c = cut.first; c < cut.first + cut.count; ++c) {
      const int64_t end = __ldg(&a.chunks[c + 1].pos);
      float acc = 0.f;
#pragma unroll 4
      for (int64_t k = __ldg(&a.chunks[c].pos); k < end; ++k) {
        const int32_t id = a.idx ? __ldg(a.idx + k) : 0;
        const int32_t e = a.perm ? __ldg(a.perm + k) : (int32_t)k;  // the edge's position in the CSR
        const float y = a.Y ? __ldg(a.Y + (a.edge_cols == 1 ? (int64_t)e : (int64_t)e * a.F + f)) : 1.f;
        const float x = a.bin == kCopyRhs ? 0.f : gathered(a, id, f);
        if (a.gradient) {  // of the vertex features: x is dO, selected where its arg names this edge
          if (a.arg && __ldg(a.arg + (int64_t)id * a.F + f) != e) continue;
          acc += a.bin == kMul ? x * y : a.bin == kDiv ? x * d_dx<kDiv>(y) : x;
        } else if (a.red == kSum) {
          if (a.w) acc = fmaf(__ldg(a.w + k), x, acc);
          else acc += message_of(a.bin, x, y);
        } else {
          const float m = message_of(a.bin, x, y);
          if (a.red == kMax) {
            if (a.arg_out) take_better<kMax>(best, at, m, e);
            else if (m > best) best = m;
          } else {
            if (a.arg_out) take_better<kMin>(best, at, m, e);
            else if (m < best) best = m;
          }
        }
      }
      group += acc;
      if ((c - cut.first) % kGroup == kGroup - 1) {
        total += group;
        group = 0.f;
      }
    }
    total += group;
    if (a.red != kSum && !a.gradient) {
      a.out[o] = best;
      if (a.arg_out) a.arg_out[o] = at;
    } else {
      float scale = 1.f;
      if (a.mean_ptr) {
        const int64_t len = __ldg(a.mean_ptr + cut.row + 1) - __ldg(a.mean_ptr + cut.row) + a.mean_self;
        scale = 1.0f / (float)len;
      }
      a.out[o] += total * scale;
    }
  }
}

}  // namespace

dg_status_t add_pieces(const Graph* g, const Plan& plan, PieceArgs a, cudaStream_t s) {
  a.chunks = plan.chunks;
  a.cuts = plan.cuts;
  a.totals = plan.totals;
  a.max_cuts = (int32_t)plan.max_cuts;
  // the number of cut rows may still be on its way to the host: the kernel reads it on the device
  int64_t blocks = plan.cut_rows >= 0 ? plan.cut_rows : plan.max_cuts;
  if (blocks > (int64_t)g->sm_count * 64) blocks = (int64_t)g->sm_count * 64;
  pieces_kernel<<<dim3((unsigned)blocks, (unsigned)((a.F + 31) / 32)), 32, 0, s>>>(a);
  DG_CUDA(cudaGetLastError());
  count_launches(1);
  return DG_OK;
}

}  // namespace dg
