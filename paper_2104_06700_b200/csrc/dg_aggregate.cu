// Host side of the aggregation: chooses the launch shape of one call (vector width, feature
// slices, source blocks), runs one launch per source block and joins the rows the plan cut.  The
// kernels are in dg_aggregate_kernels.cuh; this file compiles them for graphs without implicit self
// loops, dg_aggregate_self.cu for the others (the translation units compile side by side).
#include "dg_aggregate_kernels.cuh"

namespace dg {
namespace {

// Adds the slots of every cut row to what the row's first chunk stored.  A block takes one row and 128
// features; its 8 warps take every eighth slot, and their sums are added in warp order.  The traffic is
// one row of F floats per chunk of up to 1024 gathered rows; the launch itself is most of the cost.
// HUB: a warp adds kJoinChain slots before it adds to its total.  A small graph's chunks are short, and a hub has tens of
// thousands of them (4 M entries of a row, chunks of 96: relative error 1.0e-6 in one chain, 1.9e-7 so).  Compiled apart,
// for plans with rows of over kJoinShare slots: the loops around the loop cost every short row half a microsecond (65 k
// edges, F = 64, forward + backward 19.6 -> 20.5 us; 1.2 M, F = 47 75.6 -> 77.3).
constexpr int kJoinChain = 32, kJoinShare = kJoinChain * kWarpsPerBlock;
template <bool HUB>
__global__ void __launch_bounds__(kBlock)
join_kernel(const Chunk* __restrict__ chunks, const CutRow* __restrict__ cuts,
            const int32_t* __restrict__ totals, int32_t max_cuts, const float* __restrict__ partial, int32_t F,
            float* __restrict__ Y) {
  __shared__ float part[kWarpsPerBlock][128];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int f0 = blockIdx.y * 128;
  cudaGridDependencySynchronize();
  const int cut_rows = min(__ldg(totals + 1), max_cuts);
  for (int i = blockIdx.x; i < cut_rows; i += gridDim.x) {
    const CutRow cut = cuts[i];
    float total[4] = {0.f, 0.f, 0.f, 0.f};
    for (int k0 = warp; k0 < cut.count; k0 += kJoinShare) {
      float sum[4] = {0.f, 0.f, 0.f, 0.f};
      const int k1 = HUB ? min(cut.count, k0 + kJoinShare) : cut.count;
      for (int k = k0; k < k1; k += kWarpsPerBlock) {
        const float* p = partial + (size_t)__ldg(&chunks[cut.first + k].slot) * (size_t)F;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const int f = f0 + 32 * j + lane;
          if (f < F) sum[j] += p[f];
        }
      }
#pragma unroll
      for (int j = 0; j < 4; ++j) total[j] += sum[j];
      if (!HUB) break;
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) part[warp][32 * j + lane] = total[j];
    __syncthreads();
    const int f = f0 + threadIdx.x;
    if (threadIdx.x < 128 && f < F) {
      float t = part[0][threadIdx.x];
#pragma unroll
      for (int w = 1; w < kWarpsPerBlock; ++w) t += part[w][threadIdx.x];
      Y[(size_t)cut.row * (size_t)F + f] += t;
    }
    __syncthreads();
  }
}

// out[r][0..ld) = in[r][0..F) followed by zeros, elements of T; a thread writes 16 bytes.  Reads and
// writes are streams: bound by DRAM where the matrix exceeds L2 (561 MB of fp32 in 185 us, 6.1 TB/s read + written).
// With mean_ptr (T = float) the rows are divided by their lengths there (+ mean_self).
template <typename T>
__global__ void __launch_bounds__(256)
pad_rows_kernel(const T* __restrict__ in, int32_t F, int32_t ld, int64_t n, const int64_t* __restrict__ mean_ptr,
                int mean_self, uint4* __restrict__ out) {
  cudaTriggerProgrammaticLaunchCompletion();
  constexpr int kPer = 16 / sizeof(T);
  const uint32_t per_row = (uint32_t)ld / kPer;
  const int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x;
  const int64_t r = i / per_row;
  if (r >= n) return;
  const int f = (int)(i - r * per_row) * kPer;
  const T* src = in + r * F + f;
  union { T t[kPer]; uint4 v; } u;
#pragma unroll
  for (int q = 0; q < kPer; ++q) u.t[q] = f + q < F ? src[q] : T(0);
  if constexpr (sizeof(T) == 4) {
    if (mean_ptr) {
      const int64_t len = __ldg(mean_ptr + r + 1) - __ldg(mean_ptr + r) + mean_self;
      const float inv = len > 0 ? 1.0f / (float)len : 0.f;
#pragma unroll
      for (int q = 0; q < kPer; ++q) u.t[q] *= inv;
    }
  }
  out[i] = u.v;
}

}  // namespace

dg_status_t launch_plain(const ApArgs& a, int vec, int slices, cudaStream_t s) {
  return dispatch_type<false>(a, SelfArgs{}, vec, slices, s);
}

float* take_partial(const Graph* g, const Plan& plan, int64_t floats_per_slot, cudaStream_t s, bool* missing) {
  void* p = nullptr;
  const int64_t slots = plan.slots >= 0 ? plan.slots : plan.max_slots;
  *missing = slots > 0 && scratch_alloc(g, (size_t)slots * (size_t)floats_per_slot * sizeof(float), s, &p) != cudaSuccess;
  return static_cast<float*>(p);
}

dg_status_t join_cut_rows(const Graph* g, const Plan& plan, const float* partial, int32_t F, float* Y,
                          cudaStream_t s) {
  // the number of cut rows may still be on its way to the host: the kernel reads it on the device
  int64_t blocks = plan.cut_rows >= 0 ? plan.cut_rows : plan.max_cuts;
  if (blocks > (int64_t)g->sm_count * 64) blocks = (int64_t)g->sm_count * 64;
  const dim3 grid((unsigned)blocks, (unsigned)((F + 127) / 128));
  auto kernel = plan.most_pieces >= 0 && plan.most_pieces <= kJoinShare ? join_kernel<false> : join_kernel<true>;
  DG_CUDA(launch_kernel(kernel, grid, kBlock, s, true, (const Chunk*)plan.chunks, (const CutRow*)plan.cuts,
                        (const int32_t*)plan.totals, (int32_t)plan.max_cuts, partial, F, Y));
  count_launches(1);
  return DG_OK;
}

// Bytes of L2 one row slice of `slice` elements of `eb` bytes occupies (`F` from one row to the next): L2
// allocates 128-byte lines, and a slice that does not start on a line boundary in every row touches one
// more line; whole rows follow one another without gaps.
static double slice_footprint(int64_t F, int64_t slice, int eb) {
  if (slice >= F) return (double)(F * eb);
  const int64_t bytes = slice * eb;
  const bool aligned = (F * eb) % 128 == 0 && bytes % 128 == 0;
  return (double)(((bytes + 127) / 128) * 128 + (aligned ? 0 : 128));
}

// Whether a call first copies X into padded rows: 16-byte loads need rows that start on 16 bytes, and a
// width like 47 or 602 (8-byte rows, or 4-byte rows in bf16) otherwise gathers every row with two to
// four times as many, narrower loads.  The copy costs about two passes over X against nnz / n gathers of
// every row.  It pays from a mean degree of about 20 on, and from 8 on where it is the odd rows of over
// 128 floats that would take several times the slices (`vec` is the width X allows); rows of up to 4
// elements gain nothing, and its launch and its scratch cost more than the narrow loads of a call that
// gathers fewer than kPadMinWork elements.  Measured, us of a forward and a backward pass with / without:
// degree 50, 0.6 M edges, F = 47 57 / 58, 225 113 / 191, 602 250 / 300, 602 in bf16 215 / 287; degree
// 14.5, 1.6 M edges, F = 47 132 / 120, 110 197 / 156, 225 336 / 406, 602 849 / 672; 10 k edges, F = 41
// 27 / 19.  At degree 492, F = 602: 32.8 / 34.9 ms.
constexpr int64_t kPadMinDegree = 20, kPadMinDegreeOdd = 8, kPadMinWork = 1 << 24;
constexpr size_t kPadMaxBytes = (size_t)4 << 30;  // the pool keeps this much
bool worth_padding(const Graph* g, int32_t F, int elem_bytes, int vec) {
  const int64_t degree = vec == 1 && F > 128 ? kPadMinDegreeOdd : kPadMinDegree;
  return vec * elem_bytes < 16 && F > 4 && g->nnz >= degree * g->n && g->nnz * F >= kPadMinWork &&
         (size_t)g->n * (size_t)(F + 128 / elem_bytes) * (size_t)elem_bytes <= kPadMaxBytes;
}

// Whether the backward pass of the mean on an unweighted graph divides the rows of dOut in such a copy (also
// when they need no padding) and runs the kernel without edge factors.  That kernel reads 4 bytes less per
// edge and takes about 10 % less time; the copy is 8 bytes per element against nnz / n gathers of 4, so it
// wants long rows.  Copy and kernel: degree 492, F = 602 16.9 -> 14.9 ms, F = 256 6.7 -> 5.9 ms; degree 422,
// F = 64 565 -> 513 us; degree 85, 3.4 M edges, F = 128 162 -> 125 us.
constexpr int64_t kDivideMinDegree = 64;
static bool worth_dividing(const Graph* g, int32_t F) {
  return g->nnz >= kDivideMinDegree * g->n && g->nnz * F >= kPadMinWork &&
         (size_t)g->n * (size_t)(F + 32) * 4 <= kPadMaxBytes;
}

// Makes the copy; *copy stays nullptr when there is no memory for it (the caller then uses X as it is).
dg_status_t pad_rows(const Graph* g, const void* X, int32_t F, int elem_bytes, const int64_t* mean_ptr, int mean_self,
              cudaStream_t s, void** copy, int64_t* ld) {
  // rows of whole 32-byte sectors, of whole 128-byte lines where a row has several
  const int64_t unit = (F * elem_bytes > 512 ? 128 : 32) / elem_bytes;
  const int64_t to = (F + unit - 1) / unit * unit;
  const size_t bytes = (size_t)g->n * (size_t)to * (size_t)elem_bytes;
  if (scratch_alloc(g, bytes, s, copy) != cudaSuccess) return DG_OK;
  *ld = to;
  const unsigned blocks = (unsigned)((bytes / 16 + 255) / 256);
  if (elem_bytes == 2)
    pad_rows_kernel<uint16_t><<<blocks, 256, 0, s>>>(static_cast<const uint16_t*>(X), F, (int32_t)to, g->n, nullptr, 0,
                                                     static_cast<uint4*>(*copy));
  else
    pad_rows_kernel<float><<<blocks, 256, 0, s>>>(static_cast<const float*>(X), F, (int32_t)to, g->n, mean_ptr,
                                                  mean_self, static_cast<uint4*>(*copy));
  if (const cudaError_t e = cudaGetLastError()) {
    pool_free(*copy, s);
    *copy = nullptr;
    return cuda_fail(e, "padded copy");
  }
  count_launches(1);
  return DG_OK;
}

// Chooses the launch shape, then runs one launch per source block.
//   vector width: 16-byte loads of the gathered matrix when its rows and its base are 16-byte aligned,
//     or of its padded copy; else 8 or 4 bytes;
//   slice: 32 vectors, one per lane (512 bytes of a row), where the rows are long enough (24 entries) to
//     pay for reading the indices once per slice and F fills the slices, else 64.  Several rows of a
//     gather then cover few L2 sets' worth of one matrix at a time, and a lane keeps more edges in
//     flight.  Forward sum, F = 256, widths 256 / 128 / 64 / 32: 25 M edges, mean degree 50: 1.91 / 1.67 /
//     1.76 / 2.67 ms; 8 M edges, degree 14.5: 366 / 466 / 746 / 1354 us.  Slices narrow enough to keep
//     a graph of short rows in L2 were slower on every graph tried (12 M edges, degree 50, F = 256,
//     245 MB: 44 floats a slice 1.22 ms, 128 floats 0.73);
//   source blocks (Algorithm 2 of the paper, with L2 in the role of the CPU cache): when one
//     slice of X over all n rows exceeds the L2 budget and the segments carry split pointers,
//     the neighbour ids are cut into 2, 4, 8 or 16 ranges and each range is a launch of its
//     own, so that the rows of X a launch gathers stay L2-resident; later launches add to Y.
dg_status_t aggregate_run(const Graph* g, const ApArgs& a0, const SelfArgs& sa0, const Plan& plan,
                          const int32_t* split, cudaStream_t s) {
  ApArgs a = a0;
  SelfArgs sa = sa0;
  if (a.n == 0) return DG_OK;
  const uintptr_t px = (uintptr_t)a.X, py = (uintptr_t)a.Y;
  const bool bf16 = a.x_bf16 != 0;
  const int eb = bf16 ? 2 : 4;
  const int wide = 16 / eb;  // elements of a 16-byte load
  if (bf16 && (a.F % 2 != 0 || px % 4 != 0 || py % 8 != 0)) {
    set_error("bf16 feature matrices need an even F and 4-byte (input) / 8-byte (output) alignment");
    return DG_ERR_UNSUPPORTED;
  }
  int vec = 1;  // elements per lane and vector
  if (a.F % wide == 0 && px % 16 == 0 && py % 16 == 0) vec = wide;
  else if (bf16 && a.F % 4 == 0 && px % 8 == 0 && py % 16 == 0) vec = 4;
  else if (bf16 || (a.F % 2 == 0 && px % 8 == 0 && py % 8 == 0)) vec = 2;
  int64_t ld = a.F;
  void* padded = nullptr;
  const bool divide = worth_dividing(g, a.F) && a.mean_factors && !bf16;
  if (divide || worth_padding(g, a.F, eb, vec))
    if (dg_status_t st = pad_rows(g, a.X, a.F, eb, divide ? g->rowptr : nullptr, sa.self_ptr != nullptr, s, &padded,
                                  &ld))
      return st;
  if (padded) {
    if (divide) {  // the factors are in the copy, the own rows' too
      a.w = nullptr;
      sa.self_mean = 0;
    }
    a.X = padded;
    a.overlap = 1;
    vec = wide;
    a.narrow_store = a.F % 4 != 0 || py % 16 != 0 || (bf16 && a.F % 8 != 0);
  }
  a.row_bytes = (uint32_t)(ld * eb);

  const double budget = (double)g->l2_budget_bytes;
  const double avg_len = (double)g->nnz / (double)a.n;
  a.long_rows = avg_len >= 24.0;
  const int64_t cap = 128LL * vec;
  int64_t slice;
  int nb = 1;
  if (g->slice_features > 0) {
    slice = g->slice_features < cap ? g->slice_features : cap;
    if (slice > a.F) slice = a.F;
  } else {
    slice = a.long_rows && 2 * a.F >= 96LL * vec ? 32LL * vec : 64LL * vec;
    if (slice > a.F) slice = a.F;
  }
  if (g->source_blocks > 0) {
    nb = split ? (int)g->source_blocks : 1;
  } else if (split && g->slice_features <= 0 && (double)a.n * slice_footprint(ld, ld, eb) > budget) {
    // A width is feasible when some block count keeps one block of the slice inside the budget and
    // leaves a row at least 32 edges per block on average.  Among those, the least traffic beside the
    // gather: every slice reads the index stream again, every block after the first reads and writes
    // the output again.
    const double stream = (double)g->nnz * (a.w ? 8.0 : 4.0), output = (double)a.n * a.F * 4.0;
    double best = 0.0;
    for (int64_t wide = 64LL * vec; wide >= 8LL * vec; wide /= 2) {
      const int64_t w = wide < a.F ? wide : ld;
      int cand = 1;
      while (cand < kFineBlocks && (double)a.n / cand * slice_footprint(ld, w, eb) > budget) cand *= 2;
      if ((double)a.n / cand * slice_footprint(ld, w, eb) > budget || avg_len / cand < 32.0) continue;
      const double cost = stream * (double)((a.F + w - 1) / w) + output * (2 * cand - 1);
      if (best == 0.0 || cost < best) {
        best = cost;
        slice = w;
        nb = cand;
      }
    }
  }
  slice = slice < a.F ? (slice / vec) * vec : ld;  // a padded row ends in a vector that reaches beyond F
  if (slice < vec) slice = vec;
  if ((a.F + slice - 1) / slice > 65535) {  // grid.y limit: widen a (requested) tiny slice
    slice = (a.F + 65534) / 65535;
    slice = ((slice + vec - 1) / vec) * vec;
  }
  // even out the slices: same count, smallest width that covers F (in whole lines when X is padded)
  const int64_t nsl = (a.F + slice - 1) / slice;
  const int64_t unit = padded && nsl > 1 ? 128 / eb : vec;
  int64_t even = (a.F + nsl - 1) / nsl;
  even = ((even + unit - 1) / unit) * unit;
  if (even <= slice) slice = even;
  a.slice_f = (int32_t)slice;
  const int slices = (int)((a.F + slice - 1) / slice);

  a.chunks = plan.chunks;
  a.chunk_count = (int32_t)plan.count;
  a.few_blocks = plan.count * slices <= 4 * (int64_t)g->sm_count * 4 * kWarpsPerBlock;  // four waves
  bool missing = false;
  a.partial = take_partial(g, plan, a.F, s, &missing);
  dg_status_t st = DG_OK;
  const int per = kFineBlocks / nb;
  for (int j = 0; j < nb && st == DG_OK; ++j) {
    if (nb > 1) {
      a.seg_lo = split + (size_t)(j * per) * (size_t)a.n;
      a.seg_hi = split + (size_t)((j + 1) * per) * (size_t)a.n;
      a.accumulate = j > 0;
      a.overlap = a.overlap && j == 0;
    }
    st = sa.self_ptr ? launch_with_self_loops(a, sa, vec, slices, s) : launch_plain(a, vec, slices, s);
  }
  if (a.partial) {
    if (st == DG_OK) st = join_cut_rows(g, plan, a.partial, a.F, a.Y, s);
    pool_free(a.partial, s);
  }
  if (missing && st == DG_OK) {
    PieceArgs p{};
    p.idx = a.idx;
    p.X = a.X;
    p.ldx = ld;
    p.bf16 = bf16;
    p.w = a.w;
    p.F = a.F;
    p.red = DG_RED_SUM;
    p.mean_ptr = a.mean_rows ? a.ptr : nullptr;
    p.mean_self = sa.self_ptr != nullptr;
    p.out = a.Y;
    st = add_pieces(g, plan, p, s);
  }
  pool_free(padded, s);
  return st;
}

}  // namespace dg
