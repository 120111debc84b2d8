// Aggregation kernels: out[r] = rs_r * sum_k s_k * X[idx[k]] over one segment of a CSR (forward)
// or CSC (backward) structure.  This is the pull loop of Algorithm 1 of the paper; the register
// accumulation with one store per row follows the idea of Algorithm 3, and cutting the source
// vertices into blocks whose rows of X stay L2-resident is Algorithm 2 with L2 in the role of
// the CPU cache (one launch per block, later launches adding to the output).
//
// Work decomposition
//   Every warp takes one chunk of the direction's plan (see Plan): a run of rows, or a piece of one long
//   row, with about the same number of entries as every other chunk.  It reads the indices of the
//   chunk as one contiguous stream of 32-edge batches (one edge per lane, next batch prefetched), so
//   short rows share coalesced index loads.  Lanes are spread along the feature dimension with 16-, 8-
//   or 4-byte vector loads.  When a row slice needs fewer than 32 vectors the warp is cut into groups
//   of G lanes and the groups take different edges of the same row; their partial sums are combined by
//   a fixed shuffle tree.  U load steps per lane are in flight before the first add.
//   A piece that begins inside a row goes to a slot of a scratch array; join_kernel (dg_aggregate.cu)
//   adds the slots of a row to what its first piece stored.
// With whole rows per warp (up to 31 of them, rows over 1024 entries to a block each) a warp's longest
// serial run of edges, not the amount of work, set the time of small and of skewed graphs.  Equal chunks,
// kernel time of a forward and a backward pass on B200: 1.2 M edges, rows up to 2000, F = 47: 334 -> 57 us;
// 65 k edges, F = 64: 20.7 -> 12.1 us; 81 M edges, columns up to 10^5, F = 128: 11.5 -> 10.2 ms.
// Every output element is produced by one thread per launch in an order fixed by the plan, so the
// result is deterministic and needs no atomics in either direction.
#ifndef DG_AGGREGATE_KERNELS_CUH_
#define DG_AGGREGATE_KERNELS_CUH_
#include "dg_internal.cuh"

namespace dg {
namespace {

constexpr int kWarpsPerBlock = 8;
constexpr int kBlock = kWarpsPerBlock * 32;
constexpr unsigned kFull = 0xffffffffu;

// Accumulators are fp32 vectors of VEC floats; f8 is the 8-wide one (two float4).
struct f8 { float4 lo, hi; };
template <int VEC> struct Vec;
template <> struct Vec<1> { using T = float; };
template <> struct Vec<2> { using T = float2; };
template <> struct Vec<4> { using T = float4; };
template <> struct Vec<8> { using T = f8; };

// Storage type of the gathered matrix: fp32, or bf16 (halves every gathered byte; the sums
// stay fp32).  Pack<E, VEC>::Load is what one lane loads for VEC consecutive elements.
struct F32 { static constexpr int kBytes = 4; };
struct BF16 { static constexpr int kBytes = 2; };
template <typename E, int VEC> struct Pack { using Load = typename Vec<VEC>::T; };
template <> struct Pack<BF16, 2> { using Load = uint32_t; };
template <> struct Pack<BF16, 4> { using Load = uint2; };
template <> struct Pack<BF16, 8> { using Load = uint4; };

__device__ __forceinline__ float ldg_vec(const char* p, float) {
  return __ldg(reinterpret_cast<const float*>(p));
}
__device__ __forceinline__ float2 ldg_vec(const char* p, float2) {
  return __ldg(reinterpret_cast<const float2*>(p));
}
__device__ __forceinline__ float4 ldg_vec(const char* p, float4) {
  return __ldg(reinterpret_cast<const float4*>(p));
}
__device__ __forceinline__ uint32_t ldg_vec(const char* p, uint32_t) {
  return __ldg(reinterpret_cast<const uint32_t*>(p));
}
__device__ __forceinline__ uint2 ldg_vec(const char* p, uint2) {
  return __ldg(reinterpret_cast<const uint2*>(p));
}
__device__ __forceinline__ uint4 ldg_vec(const char* p, uint4) {
  return __ldg(reinterpret_cast<const uint4*>(p));
}
// a 32-bit word holds two bf16 values: the low half is the element with the lower index
__device__ __forceinline__ float bf_lo(uint32_t x) { return __uint_as_float(x << 16); }
__device__ __forceinline__ float bf_hi(uint32_t x) { return __uint_as_float(x & 0xffff0000u); }
// 1 / (in-degree + 1) of vertex r, from the CSR row pointer
__device__ __forceinline__ float self_factor(const int64_t* self_ptr, int64_t r) {
  return 1.0f / (float)(__ldg(self_ptr + r + 1) - __ldg(self_ptr + r) + 1);
}
__device__ __forceinline__ float ld_vec(const float* p, float) { return *p; }
__device__ __forceinline__ float2 ld_vec(const float* p, float2) {
  return *reinterpret_cast<const float2*>(p);
}
__device__ __forceinline__ float4 ld_vec(const float* p, float4) {
  return *reinterpret_cast<const float4*>(p);
}
__device__ __forceinline__ f8 ld_vec(const float* p, f8) {
  f8 v;
  v.lo = *reinterpret_cast<const float4*>(p);
  v.hi = *reinterpret_cast<const float4*>(p + 4);
  return v;
}
__device__ __forceinline__ void zero(uint32_t& a) { a = 0u; }
__device__ __forceinline__ void zero(uint2& a) { a.x = a.y = 0u; }
__device__ __forceinline__ void zero(uint4& a) { a.x = a.y = a.z = a.w = 0u; }
__device__ __forceinline__ void zero(float& a) { a = 0.f; }
__device__ __forceinline__ void zero(float2& a) { a.x = a.y = 0.f; }
__device__ __forceinline__ void zero(float4& a) { a.x = a.y = a.z = a.w = 0.f; }
__device__ __forceinline__ void add(float& a, const float& v) { a += v; }
__device__ __forceinline__ void add(float2& a, const float2& v) { a.x += v.x; a.y += v.y; }
__device__ __forceinline__ void add(float4& a, const float4& v) {
  a.x += v.x; a.y += v.y; a.z += v.z; a.w += v.w;
}
__device__ __forceinline__ void zero(f8& a) { zero(a.lo); zero(a.hi); }
__device__ __forceinline__ void add(f8& a, const f8& v) { add(a.lo, v.lo); add(a.hi, v.hi); }
// Packed bf16 loads into fp32 accumulators.  Unpacking costs as many instructions as the additions, and issue bounds these
// kernels beside the gather: sm_100 adds a bf16 operand to an fp32 sum in one instruction, and multiplies and adds two
// unpacked ones in one.  The results are those of unpacking and adding, bit for bit.  28.6 M edges, F = 602, forward and
// backward of the mean 4850 -> 4590 us (17 TB/s gathered forward, of 18.5 that the SMs can take).  In fp32, where nothing
// is unpacked, pairs of additions in one instruction changed nothing.
__device__ __forceinline__ void add(float2& a, uint32_t v) {
  asm("{.reg .b16 l, h; mov.b32 {l, h}, %2; add.rn.f32.bf16 %0, l, %0; add.rn.f32.bf16 %1, h, %1;}"
      : "+f"(a.x), "+f"(a.y)
      : "r"(v));
}
__device__ __forceinline__ void add(float4& a, uint2 v) {
  float2 lo = make_float2(a.x, a.y), hi = make_float2(a.z, a.w);
  add(lo, v.x);
  add(hi, v.y);
  a = make_float4(lo.x, lo.y, hi.x, hi.y);
}
__device__ __forceinline__ void add(f8& a, uint4 v) {
  add(a.lo, make_uint2(v.x, v.y));
  add(a.hi, make_uint2(v.z, v.w));
}
__device__ __forceinline__ void fma(float2& a, float s, uint32_t v) {
  a = __ffma2_rn(make_float2(s, s), make_float2(bf_lo(v), bf_hi(v)), a);
}
__device__ __forceinline__ void fma(float4& a, float s, uint2 v) {
  float2 lo = make_float2(a.x, a.y), hi = make_float2(a.z, a.w);
  fma(lo, s, v.x);
  fma(hi, s, v.y);
  a = make_float4(lo.x, lo.y, hi.x, hi.y);
}
__device__ __forceinline__ void fma(f8& a, float s, uint4 v) {
  fma(a.lo, s, make_uint2(v.x, v.y));
  fma(a.hi, s, make_uint2(v.z, v.w));
}
__device__ __forceinline__ void fma(float& a, float s, const float& v) { a = fmaf(s, v, a); }
__device__ __forceinline__ void fma(float2& a, float s, const float2& v) {
  a.x = fmaf(s, v.x, a.x); a.y = fmaf(s, v.y, a.y);
}
__device__ __forceinline__ void fma(float4& a, float s, const float4& v) {
  a.x = fmaf(s, v.x, a.x); a.y = fmaf(s, v.y, a.y);
  a.z = fmaf(s, v.z, a.z); a.w = fmaf(s, v.w, a.w);
}
// A scaled edge with G lanes.  Two lanes (rows of 16 numbers at most) load an edge's ids and factors as often as its
// numbers and are not bound by issue: there pairs of operations only cost registers (49 M edges, F = 16, bf16, the mean's
// backward pass 446 us with them, 436 without; F = 64 955, 1003).
template <int G, typename A, typename V>
__device__ __forceinline__ void fma_edge(A& a, float s, const V& v) {
  fma(a, s, v);
}
template <int G>
__device__ __forceinline__ void fma_edge(f8& a, float s, const uint4& v) {
  if constexpr (G == 2) {
    a.lo.x = fmaf(s, bf_lo(v.x), a.lo.x); a.lo.y = fmaf(s, bf_hi(v.x), a.lo.y);
    a.lo.z = fmaf(s, bf_lo(v.y), a.lo.z); a.lo.w = fmaf(s, bf_hi(v.y), a.lo.w);
    a.hi.x = fmaf(s, bf_lo(v.z), a.hi.x); a.hi.y = fmaf(s, bf_hi(v.z), a.hi.y);
    a.hi.z = fmaf(s, bf_lo(v.w), a.hi.z); a.hi.w = fmaf(s, bf_hi(v.w), a.hi.w);
  } else {
    fma(a, s, v);
  }
}
__device__ __forceinline__ void scale(float& a, float s) { a *= s; }
__device__ __forceinline__ void scale(float2& a, float s) { a.x *= s; a.y *= s; }
__device__ __forceinline__ void scale(float4& a, float s) { a.x *= s; a.y *= s; a.z *= s; a.w *= s; }
__device__ __forceinline__ void scale(f8& a, float s) { scale(a.lo, s); scale(a.hi, s); }
__device__ __forceinline__ float shfl_xor(float a, int m) { return __shfl_xor_sync(kFull, a, m); }
__device__ __forceinline__ float2 shfl_xor(float2 a, int m) {
  return make_float2(__shfl_xor_sync(kFull, a.x, m), __shfl_xor_sync(kFull, a.y, m));
}
__device__ __forceinline__ float4 shfl_xor(float4 a, int m) {
  return make_float4(__shfl_xor_sync(kFull, a.x, m), __shfl_xor_sync(kFull, a.y, m),
                     __shfl_xor_sync(kFull, a.z, m), __shfl_xor_sync(kFull, a.w, m));
}
__device__ __forceinline__ f8 shfl_xor(f8 a, int m) {
  f8 r;
  r.lo = shfl_xor(a.lo, m);
  r.hi = shfl_xor(a.hi, m);
  return r;
}
__device__ __forceinline__ void unpack(float (&t)[1], float v) { t[0] = v; }
__device__ __forceinline__ void unpack(float (&t)[2], float2 v) { t[0] = v.x; t[1] = v.y; }
__device__ __forceinline__ void unpack(float (&t)[4], float4 v) {
  t[0] = v.x; t[1] = v.y; t[2] = v.z; t[3] = v.w;
}
__device__ __forceinline__ void unpack(float (&t)[8], f8 v) {
  t[0] = v.lo.x; t[1] = v.lo.y; t[2] = v.lo.z; t[3] = v.lo.w;
  t[4] = v.hi.x; t[5] = v.hi.y; t[6] = v.hi.z; t[7] = v.hi.w;
}
__device__ __forceinline__ void stcs_vec(float* p, float v) { __stcs(p, v); }
__device__ __forceinline__ void stcs_vec(float* p, float2 v) { __stcs(reinterpret_cast<float2*>(p), v); }
__device__ __forceinline__ void stcs_vec(float* p, float4 v) { __stcs(reinterpret_cast<float4*>(p), v); }
__device__ __forceinline__ void stcs_vec(float* p, f8 v) {
  __stcs(reinterpret_cast<float4*>(p), v.lo);
  __stcs(reinterpret_cast<float4*>(p + 4), v.hi);
}
// Loads the neighbour id and the per-edge factor of the edge at position b + lane of the
// index stream (neutral values at or beyond `end`).
template <bool SCALED>
__device__ __forceinline__ void load_batch(const ApArgs& a, int64_t b, int end, int lane,
                                           int32_t& u, float& s) {
  u = 0;
  s = 0.f;
  const int64_t k = b + lane;
  if (k < end) {
    u = __ldcs(a.idx + k);
    if (SCALED) s = __ldcs(a.w + k);
  }
}

template <int VEC, int G, int CPL>
struct Shape {
  static constexpr int NG = 32 / G;  // edges one warp-wide load instruction covers
  // load steps in flight per lane (fewer when a step is several vectors wide), and no more
  // steps than one 32-edge batch holds
  static constexpr int U0 = CPL == 1 ? 8 : (CPL == 2 ? 4 : (VEC <= 2 && CPL == 4 ? 4 : 2));
  static constexpr int U = (U0 * NG > 32) ? (32 / NG) : U0;
};

// Adds the edges held in lanes [s, e) of the current batch (cur_u / cur_s: one edge per lane)
// into acc.  Lane group `grp` takes edges s+grp, s+grp+NG, ..., with kIds (below) U neighbouring ones of every full
// step.  Full steps of U*NG edges run without predicates; the ragged end runs once with predicated loads.  xrow[c]
// is the address of this lane's c-th vector inside row 0 of X.
template <typename E, int VEC, int G, int CPL, bool SCALED, bool STAGE>
__device__ __forceinline__ void add_edges(const char* const (&xrow)[CPL], uint32_t row_bytes,
                                          int32_t cur_u, float cur_s, int s, int e, int grp,
                                          typename Vec<VEC>::T (&acc)[CPL], uint2* stage) {
  using V = typename Pack<E, VEC>::Load;  // as loaded; unpacked while adding
  constexpr int NG = Shape<VEC, G, CPL>::NG;
  constexpr int U = Shape<VEC, G, CPL>::U;
  int p = s;
  // With one vector per lane (8 steps in flight) the edge factors are fetched while adding, so
  // that they hold no registers during the loads: that regime lives on occupancy.  With wider
  // lanes (4 or 2 steps) they are fetched with the loads and the adds do not wait for a shuffle.
  constexpr bool kLate = CPL == 1;
  // Scaled, wide lanes, source-blocked (L2-resident) passes: the batch's (id, factor) pairs go
  // through shared memory, so that one 8-byte broadcast load per step replaces two shuffles:
  // fewer wavefronts on the load/store pipe, which is what bounds that case (Reddit-like
  // backward 20.0 -> 19.3 ms).  Passes with short row pieces lose more on the extra store and
  // warp barriers per call than they gain (Products-like F = 256: 14.0 -> 16.0 ms), so the
  // passes without source blocks keep the shuffles.
  constexpr bool kStaged = SCALED && !kLate && STAGE;
  if (kStaged) {
    __syncwarp();
    stage[threadIdx.x & 31] = make_uint2((uint32_t)cur_u, __float_as_uint(cur_s));
    __syncwarp();
  }
  // Unscaled source-blocked passes with one vector per lane: the batch's ids through shared memory, so that a 16-byte
  // broadcast load replaces four shuffles (a batch begins at the piece, so steps are aligned; a lane group takes U
  // neighbouring edges then).  114.6 M edges, F = 602, forward and backward 30 300 -> 29 770 us.
  constexpr bool kIds = STAGE && kLate && !SCALED && U % 4 == 0;
  if (kIds) {
    __syncwarp();
    reinterpret_cast<uint32_t*>(stage)[threadIdx.x & 31] = (uint32_t)cur_u;
    __syncwarp();
  }
  for (; p + U * NG <= e; p += U * NG) {
    V v[U][CPL];
    float sc[kLate ? 1 : U];
    uint32_t ids[kIds ? U : 1];
    if (kIds) {
#pragma unroll
      for (int j = 0; j < U; j += 4) {
        const uint4 q = *reinterpret_cast<const uint4*>(reinterpret_cast<const uint32_t*>(stage) + p + grp * U + j);
        ids[j] = q.x; ids[j + 1] = q.y; ids[j + 2] = q.z; ids[j + 3] = q.w;
      }
    }
#pragma unroll
    for (int j = 0; j < U; ++j) {
      const int src = p + j * NG + grp;
      uint32_t u;
      if (kIds) {
        u = ids[j];
      } else if (kStaged) {
        const uint2 us = stage[src];
        u = us.x;
        sc[j] = __uint_as_float(us.y);
      } else {
        u = (uint32_t)__shfl_sync(kFull, cur_u, src);
        if (SCALED && !kLate) sc[j] = __shfl_sync(kFull, cur_s, src);
      }
      const uint64_t off = (uint64_t)u * row_bytes;
#pragma unroll
      for (int c = 0; c < CPL; ++c) v[j][c] = ldg_vec(xrow[c] + off, V());
    }
#pragma unroll
    for (int j = 0; j < U; ++j) {
      float sj = 1.f;
      if (SCALED) sj = kLate ? __shfl_sync(kFull, cur_s, p + j * NG + grp) : sc[j];
#pragma unroll
      for (int c = 0; c < CPL; ++c) {
        if (SCALED) fma_edge<G>(acc[c], sj, v[j][c]);
        else add(acc[c], v[j][c]);
      }
    }
  }
  if (p < e) {
    V v[U][CPL];
#pragma unroll
    for (int j = 0; j < U; ++j) {
      const int src = p + j * NG + grp;
      const uint32_t u = (uint32_t)__shfl_sync(kFull, cur_u, src & 31);
      const uint64_t off = (uint64_t)u * row_bytes;
#pragma unroll
      for (int c = 0; c < CPL; ++c) {
        if (src < e) v[j][c] = ldg_vec(xrow[c] + off, V());
        else zero(v[j][c]);  // an absent edge adds zeros (times whatever factor its lane holds)
      }
    }
#pragma unroll
    for (int j = 0; j < U; ++j) {
      const int src = p + j * NG + grp;
      float sj = SCALED ? __shfl_sync(kFull, cur_s, src & 31) : 1.f;
      if (SCALED && src >= e) sj = 0.f;  // lanes past the batch hold neutral factors, not NaNs
#pragma unroll
      for (int c = 0; c < CPL; ++c) {
        if (SCALED) fma_edge<G>(acc[c], sj, v[j][c]);
        else add(acc[c], v[j][c]);
      }
    }
  }
}

// Sums the partial results of the lane groups into group 0 (fixed tree).
template <int VEC, int G, int CPL>
__device__ __forceinline__ void combine_groups(typename Vec<VEC>::T (&acc)[CPL]) {
#pragma unroll
  for (int off = G; off < 32; off <<= 1) {
#pragma unroll
    for (int c = 0; c < CPL; ++c) add(acc[c], shfl_xor(acc[c], off));
  }
}

template <typename E, int VEC, int G, int CPL, bool SCALED, bool SEG, bool SELF>
__device__ __forceinline__ void ap_body(const ApArgs& a, const SelfArgs sa) {
  using V = typename Vec<VEC>::T;
  __shared__ __align__(16) uint2 stage_all[kWarpsPerBlock][32];
  // where row 0 of the warp's output would lie; in shared memory because only the store step needs it
  // and the summing loop is short of registers
  __shared__ float* out_all[kWarpsPerBlock];
  uint2* stage = stage_all[threadIdx.x >> 5];
  const int lane = threadIdx.x & 31;
  const int grp = lane / G;
  const int c0 = lane % G;
  const int f0 = blockIdx.y * a.slice_f;
  const int fend = min(a.F, f0 + a.slice_f);
  const int width = fend - f0;
  const int chunks = (width + VEC - 1) / VEC;  // the last vector of a padded X may reach beyond F
  const uint32_t row_bytes = a.row_bytes;

  // The shuffle tells the compiler that the warp's number, and with it everything read from the plan and
  // every loop bound below, is the same in all lanes: they then live in uniform registers.  Without it
  // the summing loops are 8 to 30 registers short and the same kernels take 1.1 to 1.8 times as long.
  const int chunk = blockIdx.x * kWarpsPerBlock + __shfl_sync(kFull, (int)(threadIdx.x >> 5), 0);
  if (chunk >= a.chunk_count) return;
  const int4 here = __ldg(reinterpret_cast<const int4*>(a.chunks) + chunk);
  const int4 next = __ldg(reinterpret_cast<const int4*>(a.chunks) + chunk + 1);
  if (here.z >= 0 && !a.partial) return;  // add_pieces will
  const int rb = here.x;
  // the next chunk may begin inside our last row; a chunk that begins inside a row is a piece of that row
  const int nrows = here.z >= 0 ? 1 : next.x - here.x + (next.z >= 0 ? 1 : 0);
  if (lane == 0)
    out_all[threadIdx.x >> 5] = here.z >= 0 ? a.partial + ((int64_t)here.z - here.x) * (int64_t)a.F : a.Y;
  __syncwarp();

  // Lanes whose vector falls beyond the slice re-read vector 0 and never store: the summing
  // loop then needs no per-lane predicate.
  const char* xrow[CPL];
  bool cok[CPL];
#pragma unroll
  for (int c = 0; c < CPL; ++c) {
    const int ci = c0 + c * G;
    cok[c] = ci < chunks;
    xrow[c] = reinterpret_cast<const char*>(a.X) + (size_t)(f0 + (cok[c] ? ci : 0) * VEC) * E::kBytes;
  }

  // Starts a row: zero, or, on a graph with implicit self loops, the row's own input row (taken
  // by lane group 0 only, once: not in the accumulating launches of later source blocks, and not by the
  // later pieces of a cut row).  It
  // is loaded here, ahead of the row's edges, like one more gathered row; added in the store
  // step instead, the load changed the instruction schedule of the whole summing loop (Reddit-
  // like F = 602 forward: 4.44 ms per launch against 4.0 ms, with the same instruction count).
  // The own row's factor: 1, or 1/(in-degree + 1) when the edges carry the mean's tabulated
  // factors (backward mean); the forward mean scales the whole row in the store step.
  // The next row's own row is asked into L2 one row ahead (1-2.5 % on the DRAM-bound workloads,
  // whose rows are short against a DRAM round trip).  Asking for all of a warp's own rows when
  // the warp starts made the same workloads slower (Products-like F = 602 41.4 -> 51.3 ms).
  auto start_row = [&](int r, V (&acc)[CPL], bool more_rows) {
#pragma unroll
    for (int c = 0; c < CPL; ++c) zero(acc[c]);
    if constexpr (SELF) {
      if (grp == 0 && *(float* volatile*)&out_all[threadIdx.x >> 5] == a.Y && !(SEG && a.accumulate)) {
        using L = typename Pack<E, VEC>::Load;
        const float ss = (sa.self_mean && !a.mean_rows) ? self_factor(sa.self_ptr, r) : 1.0f;
        // the warp's next row will want its own row: ask it into L2 one row ahead
        if (more_rows) {
#pragma unroll
          for (int c = 0; c < CPL; ++c)
            if (cok[c])
              asm volatile("prefetch.global.L2 [%0];" ::"l"(xrow[c] + (size_t)(r + 1) * row_bytes));
        }
#pragma unroll
        for (int c = 0; c < CPL; ++c)
          if (cok[c]) fma(acc[c], ss, ldg_vec(xrow[c] + (size_t)r * row_bytes, L()));
      }
    }
  };

  // Writes one finished row, or the part of a cut row: scales by 1/length for the mean (length + 1
  // with self loops: the forward segment length is the in-degree; a part is scaled by its whole row's
  // length, read again here) and, in a later source block, adds what the earlier blocks left there.
  auto store_row = [&](int r, V (&acc)[CPL]) {
    if (lane < G) {
      float rs = 1.0f;
      if (a.mean_rows) {
        const int len = (int)(__ldg(a.ptr + r + 1) - __ldg(a.ptr + r));
        rs = SELF ? 1.0f / (float)(len + 1) : (len > 0 ? 1.0f / (float)len : 1.0f);
      }
      float* orow = *(float* volatile*)&out_all[threadIdx.x >> 5] + (size_t)r * (size_t)a.F + f0;
#pragma unroll
      for (int c = 0; c < CPL; ++c) {
        if (cok[c]) {
          float* dst = orow + (c0 + c * G) * VEC;
          if (a.mean_rows) scale(acc[c], rs);
          if (VEC > 1 && a.narrow_store) {  // X is a padded copy, the output is not padded
            const int room = min(VEC, fend - f0 - (c0 + c * G) * VEC);
            float t[VEC];
            unpack(t, acc[c]);
#pragma unroll
            for (int q = 0; q < VEC; ++q)
              if (q < room) __stcs(dst + q, SEG && a.accumulate ? dst[q] + t[q] : t[q]);
          } else {
            if (SEG && a.accumulate) add(acc[c], ld_vec(dst, V()));
            stcs_vec(dst, acc[c]);
          }
        }
      }
    }
  };

  if constexpr (SEG) {
    // Source-blocked pass: row i of this warp contributes the positions [seg_lo, seg_hi) of its
    // segment.  The pieces are not adjacent in memory, so batches start at each piece; the
    // prefetch cursor (qi, qb) runs one batch ahead of the summing loop across rows.
    int my_lo = 0, my_hi = 0;
    if (lane < nrows) {
      my_lo = max(__ldg(a.seg_lo + rb + lane), here.y);
      my_hi = min(__ldg(a.seg_hi + rb + lane), next.y);
    }
    const unsigned work = __ballot_sync(kFull, my_hi > my_lo);
    int qi = work ? __ffs(work) - 1 : 32;
    Position qb = 0, qhi = 0;
    int32_t cur_u = 0, nxt_u = 0;
    float cur_s = 0.f, nxt_s = 0.f;
    auto step_q = [&]() {
      qb += 32;
      if (qb >= qhi) {
        const unsigned rest = qi >= 31 ? 0u : (work & ~((2u << qi) - 1u));
        qi = rest ? __ffs(rest) - 1 : 32;
        if (qi < 32) {
          qb = __shfl_sync(kFull, my_lo, qi);
          qhi = __shfl_sync(kFull, my_hi, qi);
        }
      }
    };
    if (qi < 32) {
      qb = __shfl_sync(kFull, my_lo, qi);
      qhi = __shfl_sync(kFull, my_hi, qi);
      load_batch<SCALED>(a, qb, qhi, lane, cur_u, cur_s);
      step_q();
      if (qi < 32) load_batch<SCALED>(a, qb, qhi, lane, nxt_u, nxt_s);
    }
    for (int i = 0; i < nrows; ++i) {
      const Position lo = __shfl_sync(kFull, my_lo, i);
      const Position hi = __shfl_sync(kFull, my_hi, i);
      V acc[CPL];
      start_row(rb + i, acc, i + 1 < nrows);
      for (Position b = lo; b < hi; b += 32) {
        add_edges<E, VEC, G, CPL, SCALED, SEG>(xrow, row_bytes, cur_u, cur_s, 0, (int)min(hi - b, 32u), grp, acc,
                                               stage);
        cur_u = nxt_u;
        cur_s = nxt_s;
        if (qi < 32) {
          step_q();
          if (qi < 32) load_batch<SCALED>(a, qb, qhi, lane, nxt_u, nxt_s);
        }
      }
      combine_groups<VEC, G, CPL>(acc);
      store_row(rb + i, acc);
    }
  } else {
    int my_ptr = lane <= nrows ? (int)__ldg(a.ptr + rb + lane) : 0;
    if (lane == 0) my_ptr = here.y;
    if (lane == nrows) my_ptr = next.y;
    const int stream_end = next.y;
    int b = here.y;
    int32_t cur_u, nxt_u;
    float cur_s, nxt_s;
    load_batch<SCALED>(a, b, stream_end, lane, cur_u, cur_s);
    load_batch<SCALED>(a, (int64_t)b + 32, stream_end, lane, nxt_u, nxt_s);
    for (int i = 0; i < nrows; ++i) {
      const int lo = __shfl_sync(kFull, my_ptr, i);
      const int hi = __shfl_sync(kFull, my_ptr, i + 1);
      V acc[CPL];
      start_row(rb + i, acc, i + 1 < nrows);
      int p = lo;
      while (p < hi) {
        if (p - b >= 32) {  // the stream is contiguous, so this is exactly one batch ahead
          b += 32;
          cur_u = nxt_u;
          cur_s = nxt_s;
          load_batch<SCALED>(a, (int64_t)b + 32, stream_end, lane, nxt_u, nxt_s);
        }
        const int e = min(hi - b, 32);
        add_edges<E, VEC, G, CPL, SCALED, SEG>(xrow, row_bytes, cur_u, cur_s, p - b, e, grp, acc, stage);
        p = b + e;
      }
      combine_groups<VEC, G, CPL>(acc);
      store_row(rb + i, acc);
    }
  }
}

// BLOCKS blocks per SM.  Six (40 registers): three to eight blocks are within 5 % of each other on every large
// workload (the gather is what they wait for, not the register file), six is the best for most.  Four (64
// registers) on grids of up to four waves of those: latency is the limit there, and with 40 registers not all
// of a lane's eight loads are in flight (forward + backward, kernels: 40 k edges, F = 256: 29.1 -> 21.3 us; 184 k,
// F = 256, bf16: 27.2 -> 24.7; 619 k, F = 100: 42.7 -> 39.1 of two waves or more; but 125 k, F = 48, bf16:
// 17.9 -> 20.6: a loss accepted for a rule on the grid alone; a bound below it, of one wave, would have given up the
// 619 k case).  At eight waves the two are equal.
// Three with four vectors per lane (only "slice_features" asks for such slices): the sums alone take up to 32 registers,
// and 40 spill up to 0.7 KB (F = 602 in slices of 1024, bf16: 7.9 M edges 2507 us, so 881; 1.1 M 443 / 192; in slices of
// 512, fp32: 1368 / 1182).
template <typename E, int VEC, int G, int CPL, bool SCALED, bool SEG, int BLOCKS>
__global__ void __launch_bounds__(kBlock, BLOCKS) ap_kernel(const ApArgs a) {
  cudaGridDependencySynchronize();            // the padded copy
  cudaTriggerProgrammaticLaunchCompletion();  // the join's blocks may wait beside the last of these
  ap_body<E, VEC, G, CPL, SCALED, SEG, false>(a, SelfArgs{});
}

// The same for graphs with implicit self loops: every row also sums its own input row.
template <typename E, int VEC, int G, int CPL, bool SCALED, bool SEG, int BLOCKS>
__global__ void __launch_bounds__(kBlock, BLOCKS) ap_kernel_self(const ApArgs a, const SelfArgs sa) {
  cudaGridDependencySynchronize();            // the padded copy
  cudaTriggerProgrammaticLaunchCompletion();  // the join's blocks may wait beside the last of these
  ap_body<E, VEC, G, CPL, SCALED, SEG, true>(a, sa);
}

template <typename E, int VEC, int G, int CPL, bool SCALED, bool SELF>
dg_status_t launch_variant(const ApArgs& a, const SelfArgs& sa, int slices, cudaStream_t s) {
  const dim3 grid((unsigned)((a.chunk_count + kWarpsPerBlock - 1) / kWarpsPerBlock), (unsigned)slices);
  const bool overlap = a.overlap;
  constexpr int kMany = CPL == 4 ? 3 : 6, kFew = CPL == 4 ? 3 : 4;
  if constexpr (SELF) {
    auto kernel = a.seg_lo ? ap_kernel_self<E, VEC, G, CPL, SCALED, true, kMany>
                  : a.few_blocks ? ap_kernel_self<E, VEC, G, CPL, SCALED, false, kFew>
                                 : ap_kernel_self<E, VEC, G, CPL, SCALED, false, kMany>;
    DG_CUDA(launch_kernel(kernel, grid, kBlock, s, overlap, a, sa));
  } else {
    auto kernel = a.seg_lo ? ap_kernel<E, VEC, G, CPL, SCALED, true, kMany>
                  : a.few_blocks ? ap_kernel<E, VEC, G, CPL, SCALED, false, kFew>
                                 : ap_kernel<E, VEC, G, CPL, SCALED, false, kMany>;
    DG_CUDA(launch_kernel(kernel, grid, kBlock, s, overlap, a));
  }
  count_launches(1);
  return DG_OK;
}

template <typename E, int VEC, bool SCALED, bool SELF>
dg_status_t dispatch_shape(const ApArgs& a, const SelfArgs& sa, int slices, cudaStream_t s) {
  if (a.n == 0) return DG_OK;
  const int chunks = ((a.slice_f < a.F ? a.slice_f : a.F) + VEC - 1) / VEC;  // vectors per row slice
  if (chunks <= 2) return launch_variant<E, VEC, 2, 1, SCALED, SELF>(a, sa, slices, s);
  if (chunks <= 4) return launch_variant<E, VEC, 4, 1, SCALED, SELF>(a, sa, slices, s);
  if (chunks <= 8) return launch_variant<E, VEC, 8, 1, SCALED, SELF>(a, sa, slices, s);
  if (chunks <= 16) return launch_variant<E, VEC, 16, 1, SCALED, SELF>(a, sa, slices, s);
  if (chunks <= 32) return launch_variant<E, VEC, 32, 1, SCALED, SELF>(a, sa, slices, s);
  // 33 to 44 vectors in half a warp, three each: of 32 lanes with two each a third would idle.  us of the forward sum and
  // the mean's backward pass, two / three each: F = 172, 1.2 M edges 78.6, 84.3 / 72.2, 74.6; 62 M 4612, 4834 / 4744, 4762;
  // 7.9 M in rows of 420 368, 338 / 314, 317; F = 136 76.3, 81.5 / 69.2, 71.4; 360, 336 / 289, 279.  48 vectors are no faster,
  // nor are rows of under 24 entries (14.5: F = 172 826, 1941 / 839, 1940).  The same with eight or four lanes for 17 to 24
  // or 9 to 12 vectors: 0.83 to 1.28 of the time, faster only in long rows.
  if constexpr (E::kBytes == 4 && VEC == 4) {
    if (chunks > 32 && chunks <= 44 && a.long_rows)
      return launch_variant<E, VEC, 16, 3, SCALED, SELF>(a, sa, slices, s);
  }
  if (chunks <= 64) return launch_variant<E, VEC, 32, 2, SCALED, SELF>(a, sa, slices, s);
  return launch_variant<E, VEC, 32, 4, SCALED, SELF>(a, sa, slices, s);
}

template <typename E, int VEC, bool SELF>
dg_status_t dispatch_scaled(const ApArgs& a, const SelfArgs& sa, int slices,
                            cudaStream_t s) {
  return a.w ? dispatch_shape<E, VEC, true, SELF>(a, sa, slices, s)
             : dispatch_shape<E, VEC, false, SELF>(a, sa, slices, s);
}

// Storage type and vector width chosen by the caller; SELF = the graph has implicit self loops
// (sa.self_ptr is set); the two cases are compiled in translation units of their own.
template <bool SELF>
dg_status_t dispatch_type(const ApArgs& a, const SelfArgs& sa, int vec, int slices,
                          cudaStream_t s) {
  if (a.x_bf16) {
    if (vec == 8) return dispatch_scaled<BF16, 8, SELF>(a, sa, slices, s);
    if (vec == 4) return dispatch_scaled<BF16, 4, SELF>(a, sa, slices, s);
    return dispatch_scaled<BF16, 2, SELF>(a, sa, slices, s);
  }
  if (vec == 4) return dispatch_scaled<F32, 4, SELF>(a, sa, slices, s);
  if (vec == 2) return dispatch_scaled<F32, 2, SELF>(a, sa, slices, s);
  return dispatch_scaled<F32, 1, SELF>(a, sa, slices, s);
}

}  // namespace
}  // namespace dg
#endif  // DG_AGGREGATE_KERNELS_CUH_
