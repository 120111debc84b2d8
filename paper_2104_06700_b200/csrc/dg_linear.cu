// The matrix products of a GraphSAGE layer on the fifth-generation tensor cores, in fp32:
//   forward   Y  = act(D (X W^T) + b)   n x K times (N x K)^T, the layer's epilogue fused
//   backward  dX = G W                  n x N times N x K
//             dW = G^T X                n rows reduced to N x K
//
// Arithmetic.  An fp32 number is the exact sum of three bf16 numbers, x = x0 + 2^-8 x1 + 2^-16 x2, each rounded from
// what the ones before leave: for every finite number, as the parts are held scaled up (unscaled, x2 of |x| < 2^-110 would fall
// below bf16's smallest).  Of the nine products of two such sums the six that matter are formed by the tensor cores, each
// exact, (0,2) (2,0) (1,1) (0,1) (1,0) (0,0) in this order, smallest first; the sum so far is scaled by 2^-8 where the parts'
// places add up to one less.  What is left out is at most 0.98 of 2^-24 |x||w|, 0.09 in the mean square.  The
// tensor cores add in fp32, but cut off where fp32 arithmetic rounds, so they only add kChunk products of a sum at a
// time: every chunk's result is read from tensor memory and added to a register with an fp32 addition.
// Infinities and NaN, whose parts are NaN, and sums that overflow give a NaN here: such an element is computed again
// with fp32 multiply-adds (sum_again).
// Errors against 64-bit sums, 2-norms, this / torch's fp32 GEMM: 245 k x 256 times 256 x 256 8.0e-8 / 2.9e-7, ReLU'd 7.7e-8 /
// 2.0e-7; summed over 245 k rows 2.8e-7 / 7.9e-7; 602 products 1.04e-7 / 4.5e-7; operands of 2^-126 7.8e-8 / 2.9e-7.  Rows with
// one to three numbers that are not 0, where the cut-off shows, 4.5e-8 to 5.6e-8 / 2.5e-8 to 3.6e-8, eight 6.5e-8 / 5.4e-8, sixteen
// 7.1e-8 / 7.4e-8.  Adding the (0,0) products apart from the others, so that their sum with the rest is an fp32 addition, gave
// 2.6e-8 for one number and took 231 us instead of 199 (all eight products above 2^-32: 2.53e-8, 254 us).
//
// Shape of the kernel.  A block computes 128 x up to 256 elements at a time, one block per SM.  The fp32 operands arrive in a
// ring of chunks in shared memory, by asynchronous copies (loads to registers need a place in the first-level cache,
// of which the operands leave a few KB: two to three times slower).  Sixteen warps split a chunk into parts, in the
// layout without swizzle (8 rows x 16 bytes, contiguous), and a seventeenth issues the matrix instructions of
// the chunk (900 to 1300 cycles, which would hold up the others).  They run while the sixteen add the chunk
// before to their sums and split the next.  The stream of chunks runs over tile borders.  The weights are split once, by a
// kernel of their own, and arrive as one bulk copy per chunk, asked for by an eighteenth warp.
//
// What bounds it, per tile of 128 x 256 and K = 256: the tensor cores, 12 300 cycles at their nominal rate of the 27 000 it
// takes; the rest is the epilogue and the chunks' chain of barriers.  245 k x 256 x 256: 189 us with the epilogue, of
// 117 for six bf16 products at the measured rate of 1640 TFLOP/s and 77 for the bytes; torch's SIMT GEMM and an elementwise
// pass 660.  The gradient of the weights is bound by shared memory, which takes every number in, splits it and feeds it out
// (2300 cycles a chunk of 768 of the tensor cores).
#include "dg_internal.cuh"

namespace dg {
namespace {

__device__ unsigned long long g_expired;  // blocks that gave up a wait

constexpr int kWorkers = 512, kWarps = kWorkers / 32, kThreads = kWorkers + 128;
constexpr int kM = 128;
constexpr int kChunk = 32;                // products of a sum per chunk: two matrix instructions per pair of parts
constexpr int kGroups = kChunk / 8;       // 16-byte groups of a row of a part
// Bytes from a group to the next: its rows, 16 bytes each, and 32 so that the writes of eight lanes, two rows in four
// groups, fall into different banks.
__host__ __device__ constexpr int group_stride(int rows) { return rows * 16 + 32; }
__host__ __device__ constexpr int operand_bytes(int rows) { return 3 * kGroups * group_stride(rows); }
constexpr int kTileBytes = 32 * 32 * 4;  // of a warp's staging tile
constexpr int kPartBits = 8;             // a part is held as 2^kPartBits times what it is to the part before

// Columns of a tile, and shared memory: two stages of operands, the ring of fp32 chunks, and staging tiles of the first
// six warps; the others' lie in a stage of A and a slot of the ring that are free when a tile of results is written.
// Without the weights' parts B goes through the ring too, and the tile is half as wide to leave room for three chunks.
template <bool SPLIT_B>
struct Shape {
  static constexpr int kN = SPLIT_B ? 256 : 128;
  static constexpr int kColumns = kN / 4;  // of a warp: four warps share the columns, four the rows
  static constexpr int kRing = 3;
  static constexpr int kRaw = (kM + (SPLIT_B ? 0 : kN)) * kChunk * 4;
  static constexpr int kB = 2 * operand_bytes(kM);
  static constexpr int kRingAt = kB + 2 * operand_bytes(kN);
  static constexpr int kTileAt = kRingAt + kRing * kRaw;
  static constexpr int kBytes = kTileAt + 6 * kTileBytes;
  static_assert(6 * kTileBytes <= operand_bytes(kM) && 4 * kTileBytes <= kRaw && kWarps == 16, "places of the tiles");
  static_assert(kBytes <= 227 * 1024 - 256, "shared memory of a block");
};

// A matrix as an operand: element (r, k), k counting along the sum, at p[r * ld + k] (ALONG) or p[k * ld + r].
struct LinearArgs {
  const float* A;
  const float* B;
  const unsigned char* image;  // B split before, see split_kernel
  int64_t lda, ldb;
  int rows_a, rows_b;       // sizes: M, N
  int depth;                // length of the sum
  int depth_slice;          // of one slice of the sum (a multiple of kChunk, or all of it: ALONG operands have one)
  int tiles_m, tiles_n, slices;
  int vector_a, vector_b;   // 16-byte copies are possible
  const float* scale;       // epilogue, each may be nullptr: of the rows
  const float* bias;        // of the columns
  int relu;
  float* out;               // slice s writes rows_a x rows_b at out + s * rows_a * rows_b
  int vector_out;
  int linear_out;           // a tile's results are one stretch of memory that fits the staging tiles
};

__device__ __forceinline__ uint32_t smem_address(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbarrier_init(uint32_t bar, int count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbarrier_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
// Waits for the phase of that parity.  Gives up after 2^22 tries, all but the first half a microsecond apart, or when
// another thread of the block has (the word at `expired`, in shared memory).  A loop without the time: the workers have no
// registers left for it.
__device__ __forceinline__ bool mbarrier_wait(uint32_t bar, uint32_t parity, uint32_t expired) {
#pragma unroll 1
  for (int i = 0; i < 1 << 22; ++i) {
    uint32_t done;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\tselp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(done) : "r"(bar), "r"(parity) : "memory");
    if (done) return true;
    if (i < 256) continue;
    asm volatile("ld.volatile.shared.u32 %0, [%1];" : "=r"(done) : "r"(expired) : "memory");
    if (done) return false;
    __nanosleep(500);
  }
  asm volatile("st.volatile.shared.u32 [%0], %1;" ::"r"(expired), "r"(1) : "memory");
  return false;
}

// Starts a copy of `bytes` (a multiple of 16) to shared memory; `bar` completes its phase when they have arrived.
__device__ __forceinline__ void bulk_copy(uint32_t to, const void* from, uint32_t bytes, uint32_t bar) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(to),
               "l"(from), "r"(bytes), "r"(bar)
               : "memory");
}

// Copies 16 or 4 bytes to shared memory, or zeros.
__device__ __forceinline__ void copy_16(uint32_t to, const float* from, bool on) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(to), "l"(from), "r"(on ? 16 : 0) : "memory");
}
__device__ __forceinline__ void copy_4(uint32_t to, const float* from, bool on) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(to), "l"(from), "r"(on ? 4 : 0) : "memory");
}

// Shared-memory descriptor of an operand without swizzle: its address, the bytes from one 16-byte group of a row to
// the next (leading offset) and from 8 rows to the next 8 (stride offset), in units of 16 bytes; bit 46: version 1.
__device__ __forceinline__ uint64_t operand(uint32_t address, int stride) {
  return (uint64_t)((address >> 4) & 0x3fff) | (uint64_t)(stride >> 4) << 16 | (uint64_t)(128 >> 4) << 32 |
         (uint64_t)1 << 46;
}
// D[128 x n] = A[128 x 16] B[n x 16]^T + D 2^-SHIFT, or without D; bf16 in, fp32 out
template <int SHIFT>
__device__ __forceinline__ void mma(uint32_t d, uint64_t a, uint64_t b, uint32_t shape, bool add) {
  if constexpr (SHIFT == 0)
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d), "l"(a), "l"(b), "r"(shape),
        "r"((uint32_t)add)
        : "memory");
  else
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p, %5;\n\t}" ::"r"(d), "l"(a), "l"(b), "r"(shape),
        "r"((uint32_t)add), "n"(SHIFT)
        : "memory");
}

// 16 columns of this warp's 32 lanes of tensor memory (32 at a time spill: seventeen warps have 96 registers)
__device__ __forceinline__ void load_accumulators(float2 (&v)[8], uint32_t address) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];\n\t"
      "tcgen05.wait::ld.sync.aligned;"
      : "=f"(v[0].x), "=f"(v[0].y), "=f"(v[1].x), "=f"(v[1].y), "=f"(v[2].x), "=f"(v[2].y), "=f"(v[3].x), "=f"(v[3].y),
        "=f"(v[4].x), "=f"(v[4].y), "=f"(v[5].x), "=f"(v[5].y), "=f"(v[6].x), "=f"(v[6].y), "=f"(v[7].x), "=f"(v[7].y)
      : "r"(address)
      : "memory");
}

__device__ __forceinline__ float max_nan(float x, float y) {
  float r;
  asm("max.NaN.f32 %0, %1, %2;" : "=f"(r) : "f"(x), "f"(y));
  return r;
}

// Two numbers rounded to bf16, the first in the low half.
__device__ __forceinline__ uint32_t round_pair(float lo, float hi) {
  uint32_t r;
  asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(r) : "f"(hi), "f"(lo));
  return r;
}
// Splits eight numbers of a row and writes the parts at `to` and every kGroups * stride bytes on.
__device__ __forceinline__ void put(unsigned char* to, int stride, const float (&x)[8]) {
  constexpr float kUp = 1 << kPartBits;  // exact: what is left is at most 2^-kPartBits of the number
  uint32_t p[3][4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    // exact but for the roundings to bf16, of which the last is exact too; two in an instruction
    float2 r = make_float2(x[2 * i], x[2 * i + 1]);
#pragma unroll
    for (int t = 0; t < 3; ++t) {
      p[t][i] = round_pair(r.x, r.y);
      r = __ffma2_rn(make_float2(__uint_as_float(p[t][i] << 16), __uint_as_float(p[t][i] & 0xffff0000u)),
                     make_float2(-1.f, -1.f), r);
      r = __fmul2_rn(r, make_float2(kUp, kUp));
    }
  }
#pragma unroll
  for (int t = 0; t < 3; ++t)
    *reinterpret_cast<uint4*>(to + t * kGroups * stride) = make_uint4(p[t][0], p[t][1], p[t][2], p[t][3]);
}

// ---- a thread's share of an operand's chunk of kM (= Shape<false>::kN) rows
// In the ring [row][k] (ALONG; a warp copies the eight rows that it splits) or [k][row].  A thread copies two quads and
// splits eight numbers of one row.
template <bool ALONG>
struct Share {
  const float* from;  // the thread's first quad at k = 0 of the tile; the second: four rows, or half a chunk, on
  int r;              // its row

  static __device__ __forceinline__ int place() { return ALONG ? threadIdx.x % 8 * 4 : threadIdx.x / (kM / 4); }
  // the tile's rows begin at r0
  __device__ __forceinline__ void begin(const float* p, int64_t ld, int r0) {
    r = r0 + (ALONG ? threadIdx.x / 32 * 8 + threadIdx.x % 32 / 8 : threadIdx.x % (kM / 4) * 4);
    from = ALONG ? p + r * ld + place() : p + place() * ld + r;
  }
  // Fetches the chunk at k0; zeros outside the matrix (rows from `rows` on) or from k_end on.  `p`: any address to name.
  __device__ __forceinline__ void copy(float* ring, int k0, int k_end, int rows, const float* p, int64_t ld,
                                       bool vector) const {
    // in quads: warp w's 64 begin at 64 w
    const uint32_t to =
        smem_address(ring) + 16 * (ALONG ? threadIdx.x / 32 * 64 + threadIdx.x % 32 : threadIdx.x);
    const float* q = from + (ALONG ? (int64_t)k0 : k0 * ld);
#pragma unroll
    for (int h = 0; h < 2; ++h, q += (ALONG ? 4 : kChunk / 2) * ld) {
      const int kk = k0 + place() + (ALONG ? 0 : kChunk / 2 * h), rr = r + (ALONG ? 4 * h : 0);
      const uint32_t at = to + h * (ALONG ? 32 : kWorkers) * 16;
      if (vector) {  // rows of whole quads
        const bool on = rr < rows && kk < k_end;
        copy_16(at, on ? q : p, on);
      } else {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const bool on = ALONG ? rr < rows && kk + i < k_end : rr + i < rows && kk < k_end;
          copy_4(at + 4 * i, on ? q + i : p, on);
        }
      }
    }
  }
};
template <bool ALONG>
__device__ __forceinline__ void split_chunk(unsigned char* parts, int stride, const float* ring, int width) {
  const int t = threadIdx.x;
  const int row = ALONG ? t / kGroups : t % kM, group = ALONG ? t % kGroups : t / kM;
  if (row >= width) return;
  float x[8];
  if (ALONG) {
    const float4 a = *reinterpret_cast<const float4*>(ring + 8 * t);
    const float4 b = *reinterpret_cast<const float4*>(ring + 8 * t + 4);
    x[0] = a.x; x[1] = a.y; x[2] = a.z; x[3] = a.w;
    x[4] = b.x; x[5] = b.y; x[6] = b.z; x[7] = b.w;
  } else {
#pragma unroll
    for (int i = 0; i < 8; ++i) x[i] = ring[(group * 8 + i) * kM + row];
  }
  put(parts + group * stride + row * 16, stride, x);
}
static_assert(kM * kGroups == kWorkers && kM == Shape<false>::kN, "shares of the threads");

template <bool ALONG>
__device__ __forceinline__ float element(const float* p, int64_t ld, int64_t r, int64_t k) {
  return __ldg(ALONG ? p + r * ld + k : p + k * ld + r);
}

// Columns of the tile at n0, in whole steps of 16.
template <int N>
__device__ __forceinline__ int tile_width(int columns, int n0) {
  return min((columns - n0 + 15) / 16 * 16, N);
}

// The tile and the part of the sum that item i of the grid's work is.
struct Item {
  int m0, n0, k0, k1, slice, chunks;
};
template <int N>
__device__ __forceinline__ Item item_of(const LinearArgs& a, int i) {
  Item t;
  t.n0 = i % a.tiles_n * N;
  i /= a.tiles_n;
  t.m0 = i % a.tiles_m * kM;
  t.slice = i / a.tiles_m;
  t.k0 = t.slice * a.depth_slice;
  t.k1 = a.depth - t.k0 > a.depth_slice ? t.k0 + a.depth_slice : a.depth;
  t.chunks = (t.k1 - t.k0 + kChunk - 1) / kChunk;
  return t;
}

__device__ __forceinline__ void sync_workers() { asm volatile("bar.sync 1, %0;" ::"n"(kWorkers) : "memory"); }
__device__ __forceinline__ bool any_worker(bool mine) {
  uint32_t any;
  asm volatile("{\n\t.reg .pred p, q;\n\tsetp.ne.u32 p, %1, 0;\n\tbar.red.or.pred q, 1, %2, p;\n\tselp.u32 %0, 1, 0, q;\n\t}"
               : "=r"(any) : "r"((uint32_t)mine), "n"(kWorkers) : "memory");
  return any != 0;
}

// The results of the block that are NaN once more with fp32 multiply-adds, in the order of the sum: infinities and NaN,
// and sums that overflow, come out as NaN above.  All workers take 128 columns of a tile at a time, eight rows and four
// columns each, through shared memory, as the inputs may be NaN throughout.
// 20 k x 256 x 256 of NaN, us: forward 252, gradient of the input 236, of the weights 117 (an element per lane 10031, 6411,
// 3640; torch 79 and 92); 245 k 1726, 1609, 1163 (torch 581, 593).
constexpr int kAgainDepth = 32, kAgainRow = kM + 4;
template <bool ALONG_A, bool ALONG_B, int kN>
__device__ __noinline__ void sum_again(const LinearArgs& a, float* space) {
  constexpr int kLoads = kAgainDepth * kM / kWorkers, kStage = 2 * kAgainDepth * kAgainRow;
  const int items = a.tiles_m * a.tiles_n * a.slices;
  const int t = threadIdx.x, tr = t / 32 * 8, tc = t % 32 * 4;
  for (int i = blockIdx.x; i < items; i += gridDim.x) {
    const Item now = item_of<kN>(a, i);
    float* out = a.out + (int64_t)now.slice * a.rows_a * a.rows_b;
    for (int n0 = now.n0; n0 < min(now.n0 + kN, a.rows_b); n0 += kM) {
      auto each = [&](auto f) {  // of the thread's results
#pragma unroll
        for (int p = 0; p < 8; ++p)
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            const int r = now.m0 + tr + p, n = n0 + tc + q;
            if (r < a.rows_a && n < a.rows_b) f(p, q, r, n, out + (int64_t)r * a.rows_b + n);
          }
      };
      bool nan = false;
      each([&](int, int, int, int, float* y) { nan = nan || *y != *y; });
      if (!any_worker(nan)) continue;
      float xa[kLoads], xb[kLoads], sum[8][4] = {};
      auto load = [&](int k) {
#pragma unroll
        for (int j = 0; j < kLoads; ++j) {
          const int ka = k + (ALONG_A ? t % 32 : t / kM + 4 * j), ra = now.m0 + (ALONG_A ? t / 32 + 16 * j : t % kM);
          const int kb = k + (ALONG_B ? t % 32 : t / kM + 4 * j), rb = n0 + (ALONG_B ? t / 32 + 16 * j : t % kM);
          xa[j] = ra < a.rows_a && ka < now.k1 ? element<ALONG_A>(a.A, a.lda, ra, ka) : 0.f;
          xb[j] = rb < a.rows_b && kb < now.k1 ? element<ALONG_B>(a.B, a.ldb, rb, kb) : 0.f;
        }
      };
      auto store = [&](float* to) {
#pragma unroll
        for (int j = 0; j < kLoads; ++j) {
          to[ALONG_A ? t % 32 * kAgainRow + t / 32 + 16 * j : (t / kM + 4 * j) * kAgainRow + t % kM] = xa[j];
          to[kStage / 2 + (ALONG_B ? t % 32 * kAgainRow + t / 32 + 16 * j : (t / kM + 4 * j) * kAgainRow + t % kM)] = xb[j];
        }
      };
      load(now.k0);
      store(space);
      sync_workers();
      int stage = 0;
#pragma unroll 1
      for (int k = now.k0; k < now.k1; k += kAgainDepth, stage ^= 1) {
        const bool more = k + kAgainDepth < now.k1;
        if (more) load(k + kAgainDepth);
        const float* from = space + stage * kStage;
#pragma unroll 4
        for (int kk = 0; kk < kAgainDepth; ++kk) {
          const float* x = from + kk * kAgainRow + tr;
          const float4 w = *reinterpret_cast<const float4*>(from + kStage / 2 + kk * kAgainRow + tc);
#pragma unroll
          for (int p = 0; p < 8; ++p) {
            sum[p][0] = fmaf(x[p], w.x, sum[p][0]);
            sum[p][1] = fmaf(x[p], w.y, sum[p][1]);
            sum[p][2] = fmaf(x[p], w.z, sum[p][2]);
            sum[p][3] = fmaf(x[p], w.w, sum[p][3]);
          }
        }
        if (more) store(space + (stage ^ 1) * kStage);
        sync_workers();
      }
      each([&](int p, int q, int r, int n, float* y) {
        if (*y == *y) return;
        const float z = fmaf(sum[p][q], a.scale ? __ldg(a.scale + r) : 1.f, a.bias ? __ldg(a.bias + n) : 0.f);
        *y = max_nan(z, a.relu ? 0.f : -INFINITY);
      });
    }
  }
}

// After a wait that ran out: the workers make the block's results NaN.
template <int kN>
__device__ __noinline__ void give_up(const LinearArgs& a) {
  if (threadIdx.x == 0) atomicAdd(&g_expired, 1ull);
  for (int i = blockIdx.x; i < a.tiles_m * a.tiles_n * a.slices; i += gridDim.x) {
    const Item t = item_of<kN>(a, i);
    float* out = a.out + ((int64_t)t.slice * a.rows_a + t.m0) * a.rows_b + t.n0;
    for (int e = threadIdx.x; e < kM * kN; e += kWorkers)
      if (t.m0 + e / kN < a.rows_a && t.n0 + e % kN < a.rows_b) out[(int64_t)(e / kN) * a.rows_b + e % kN] = NAN;
  }
}

// SPLIT_B: B has been split before (a.image).
template <bool ALONG_A, bool ALONG_B, bool SPLIT_B>
__global__ void __launch_bounds__(kThreads, 1) linear_kernel(const __grid_constant__ LinearArgs a) {
  using S = Shape<SPLIT_B>;
  constexpr int kN = S::kN;
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ uint32_t tmem_base;
  __shared__ uint64_t filled[2];   // the workers have written a stage, and read the tensor memory that it will go to
  __shared__ uint64_t done[2];     // the matrix instructions of a stage have finished
  __shared__ uint64_t arrived[2];  // a stage's chunk of the image has arrived
  __shared__ uint64_t idle;        // after a wait that ran out: no matrix instruction is in flight
  __shared__ int expired;          // a wait has run out: nothing more is started, the block's results are NaN
  __shared__ int again;            // a result has to be formed again
  __shared__ int never;            // stays 0
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int items = a.tiles_m * a.tiles_n * a.slices;
  const uint32_t filled0 = smem_address(filled), done0 = smem_address(done), arrived0 = smem_address(arrived);
  if (warp == kWarps) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_address(&tmem_base))
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  if (threadIdx.x == 0) {
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      mbarrier_init(filled0 + 8 * i, kWarps);
      mbarrier_init(done0 + 8 * i, 1);
      mbarrier_init(arrived0 + 8 * i, 1);
    }
    mbarrier_init(smem_address(&idle), 1);
    expired = never = again = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = tmem_base;
  bool good = true;
  // Chunk j of the stream, counted over all tiles: its stage is j % 2, and it completes the phases of a barrier in turn.
  // A thread waits for every phase of a barrier, in order, before the next can complete.
  auto wait_for = [&](uint32_t barriers, int j) {
    good = good && mbarrier_wait(barriers + 8 * (j & 1), j >> 1 & 1, smem_address(&expired));
  };

  // The launch gives every thread 96 registers; the workers, whose sums take 64, get 112 and the last four warps keep 24:
  // 512 x 112 + 128 x 24 = 60416 of 640 x 96 = 61440.  Spills would go to memory: no first-level cache is left.
  if (warp < kWarps) {
    // ---- the workers
    asm volatile("setmaxnreg.inc.sync.aligned.u32 112;");
    float2 acc[S::kColumns / 2];
#pragma unroll
    for (int i = 0; i < S::kColumns / 2; ++i) acc[i] = make_float2(0.f, 0.f);

    // the ring: the next chunk that is fetched, at ring_k of a sum up to ring_end
    int ring_item = blockIdx.x, ring_slot = 0, ring_k, ring_end;
    Share<ALONG_A> share_a;
    Share<ALONG_B> share_b;
    auto ring_begin = [&]() {
      const Item t = item_of<kN>(a, ring_item);
      ring_k = t.k0;
      ring_end = t.k1;
      share_a.begin(a.A, a.lda, t.m0);
      if (!SPLIT_B) share_b.begin(a.B, a.ldb, t.n0);
    };
    ring_begin();
    auto ring_next = [&]() {
      if (ring_item < items) {
        float* to = reinterpret_cast<float*>(smem + S::kRingAt + ring_slot * S::kRaw);
        share_a.copy(to, ring_k, ring_end, a.rows_a, a.A, a.lda, a.vector_a);
        if (!SPLIT_B) share_b.copy(to + kM * kChunk, ring_k, ring_end, a.rows_b, a.B, a.ldb, a.vector_b);
        ring_slot = ring_slot + 1 == S::kRing ? 0 : ring_slot + 1;
        ring_k += kChunk;
        if (ring_k >= ring_end) {
          ring_item += gridDim.x;
          if (ring_item < items) ring_begin();
        }
      }
      asm volatile("cp.async.commit_group;" ::: "memory");  // empty groups behind the last chunk keep the count
    };

    // Adds chunk j to the sums; behind a tile's last, writes the tile, whose number is `item` then and else -1.
    auto drain = [&](int j, int slot, int width, int item) {
      const int share = (width / 16 + 3) / 4 * 16;
      const int c0 = min((warp >> 2) * share, width), c1 = min(c0 + share, width);
      wait_for(done0, j);
      __syncwarp();
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const uint32_t from = tmem + ((uint32_t)(warp & 3) << 21) + (uint32_t)((j & 1) * kN + c0);
#pragma unroll
      for (int b = 0; b < S::kColumns / 16; ++b) {
        if (c0 + 16 * b >= c1) break;
        float2 v[8];
        load_accumulators(v, from + 16 * b);
#pragma unroll
        for (int i = 0; i < 8; ++i) acc[8 * b + i] = __fadd2_rn(acc[8 * b + i], v[i]);
      }
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      if (item < 0) return;
      const Item rt = item_of<kN>(a, item);
      const int row0 = rt.m0 + (warp & 3) * 32, m = row0 + lane;
      const float s = a.scale && m < a.rows_a ? __ldg(a.scale + m) : 1.f;
      float* out = a.out + (int64_t)rt.slice * a.rows_a * a.rows_b;
      const float least = a.relu ? 0.f : -INFINITY;  // act(y) = max(y, least), NaN stays NaN
      float2 check = make_float2(0.f, 0.f);          // becomes NaN if a sum is NaN or infinite
#pragma unroll
      for (int i = 0; i < S::kColumns / 2; ++i) check = __ffma2_rn(acc[i], make_float2(0.f, 0.f), check);
      if (check.x + check.y != 0.f) {
        again = 1;
#pragma unroll
        for (int i = 0; i < S::kColumns / 2; ++i) acc[i] = __ffma2_rn(acc[i], make_float2(0.f, 0.f), acc[i]);  // all NaN
      }
      // The stage of chunk j and the slot split last are free until the next chunk: 32 x 32 numbers for every warp, so that
      // results leave in whole lines (in pieces of 32 bytes, from tiles of 8 columns, this took 11 000 cycles of 26 000 a tile).
      sync_workers();
      float* tile = reinterpret_cast<float*>(
          warp < 6 ? smem + S::kTileAt + warp * kTileBytes
                   : warp < 12 ? smem + (j & 1) * operand_bytes(kM) + (warp - 6) * kTileBytes
                               : smem + S::kRingAt + slot * S::kRaw + (warp - 12) * kTileBytes);
      if (a.linear_out) {
        // Rows of a few columns that allow no vectors: written row by row they cost 20 cycles for every 16 numbers.
        float* line = reinterpret_cast<float*>(smem + S::kTileAt);
        const int N = a.rows_b;
        float* mine = line + ((warp & 3) * 32 + lane) * N + c0;
        const int cols = min(c1, N) - c0;  // at most 16
        const float bias = a.bias && lane < cols ? __ldg(a.bias + c0 + lane) : 0.f;
#pragma unroll
        for (int i = 0; i < 16; ++i) {
          const float x = i % 2 ? acc[i / 2].y : acc[i / 2].x;
          const float y = max_nan(fmaf(x, s, __shfl_sync(0xffffffffu, bias, i)), least);
          if (i < cols) mine[i] = y;
        }
        sync_workers();
        const int count = min(kM, a.rows_a - rt.m0) * N;
        float* to = out + (int64_t)rt.m0 * N;  // 128 rows on from the matrix's start: aligned as that is
        for (int i = 4 * threadIdx.x; i < count; i += 4 * kWorkers) {
          if (i + 4 <= count) *reinterpret_cast<float4*>(to + i) = *reinterpret_cast<const float4*>(line + i);
          else
            for (int k = i; k < count; ++k) to[k] = line[k];
        }
      }
#pragma unroll
      for (int b = 0; b < S::kColumns / 32; ++b) {
        if (c0 + 32 * b >= c1 || a.linear_out) break;
        const int n = rt.n0 + c0 + 32 * b, cols = min(min(32, c1 - c0 - 32 * b), a.rows_b - n);
        __syncwarp();
#pragma unroll
        for (int q = 0; q < 8; ++q) {  // quad q of row r at place q ^ r: different banks both ways
          const float2 x = acc[16 * b + 2 * q], y = acc[16 * b + 2 * q + 1];
          *reinterpret_cast<float4*>(tile + lane * 32 + ((q ^ lane) & 7) * 4) = make_float4(x.x, x.y, y.x, y.y);
        }
        __syncwarp();
        if (a.vector_out && cols % 4 == 0) {
          const int q = lane & 7, c = q * 4;
          float4 bias = make_float4(0.f, 0.f, 0.f, 0.f);
          if (a.bias && c < cols)
            bias = make_float4(__ldg(a.bias + n + c), __ldg(a.bias + n + c + 1), __ldg(a.bias + n + c + 2),
                               __ldg(a.bias + n + c + 3));
          float* to = out + (int64_t)(row0 + (lane >> 3)) * a.rows_b + n + c;
#pragma unroll 1
          for (int i = 0; i < 8; ++i, to += 4 * (int64_t)a.rows_b) {
            const int r = 4 * i + (lane >> 3);
            const float sr = __shfl_sync(0xffffffffu, s, r);
            float4 y = *reinterpret_cast<const float4*>(tile + r * 32 + ((q ^ r) & 7) * 4);
            y.x = max_nan(fmaf(y.x, sr, bias.x), least);
            y.y = max_nan(fmaf(y.y, sr, bias.y), least);
            y.z = max_nan(fmaf(y.z, sr, bias.z), least);
            y.w = max_nan(fmaf(y.w, sr, bias.w), least);
            if (row0 + r < a.rows_a && c < cols) *reinterpret_cast<float4*>(to) = y;
          }
        } else {
          const float bias = a.bias && lane < cols ? __ldg(a.bias + n + lane) : 0.f;
#pragma unroll 1
          for (int r = 0; r < 32; ++r) {
            const float sr = __shfl_sync(0xffffffffu, s, r);
            const float y = tile[r * 32 + ((lane >> 2 ^ r) & 7) * 4 + (lane & 3)];
            if (row0 + r < a.rows_a && lane < cols)
              out[(int64_t)(row0 + r) * a.rows_b + n + lane] = max_nan(fmaf(y, sr, bias), least);
          }
        }
      }
      sync_workers();
#pragma unroll
      for (int i = 0; i < S::kColumns / 2; ++i) acc[i] = make_float2(0.f, 0.f);
    };

    for (int i = 0; i < S::kRing - 1; ++i) ring_next();
    int j = 0, slot = 0, before = 0, finished = -1;  // width of the chunk before's tile, and its number if that was its last
    for (int i = blockIdx.x; i < items; i += gridDim.x) {
      const Item now = item_of<kN>(a, i);
      const int width = tile_width<kN>(a.rows_b, now.n0);
      for (int left = now.chunks; left > 0; --left, ++j) {
        asm volatile("cp.async.wait_group %0;" ::"n"(S::kRing - 2) : "memory");  // this thread's part of chunk j is there
        // A thread splits what others copied, of its warp or of any; and they are done with the slot that is filled next.
        if (SPLIT_B && ALONG_A) __syncwarp();
        else sync_workers();
        ring_next();
        // The stage is free: the chunk before the last, which had it, has been drained.
        unsigned char* pa = smem + (j & 1) * operand_bytes(kM);
        const float* raw = reinterpret_cast<const float*>(smem + S::kRingAt + slot * S::kRaw);
        const int split_slot = slot;
        slot = slot + 1 == S::kRing ? 0 : slot + 1;
        split_chunk<ALONG_A>(pa, group_stride(kM), raw, kM);
        if (!SPLIT_B)
          split_chunk<ALONG_B>(smem + S::kB + (j & 1) * operand_bytes(kN), group_stride(width), raw + kM * kChunk, width);
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncwarp();
        if (lane == 0) mbarrier_arrive(filled0 + 8 * (j & 1));
        if (j > 0) drain(j - 1, split_slot, before, finished);
        before = width;
        finished = left == 1 ? i : -1;
      }
    }
    if (j > 0) drain(j - 1, slot, before, finished);  // nothing is in the ring any more
    asm volatile("cp.async.wait_all;" ::: "memory");
    sync_workers();
    if (again) sum_again<ALONG_A, ALONG_B, kN>(a, reinterpret_cast<float*>(smem));
    } else {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 24;");
    if (warp == kWarps) {
      // ---- the issuing warp; one lane works
      if (lane == 0) {
        const uint64_t a0 = operand(smem_address(smem), group_stride(kM));
        int j = 0;
        for (int i = blockIdx.x; i < items && good; i += gridDim.x) {
          const Item now = item_of<kN>(a, i);
          const int width = tile_width<kN>(a.rows_b, now.n0), strb = group_stride(width);
          const uint64_t b0 = operand(smem_address(smem + S::kB), strb);
          // bf16 operands, fp32 accumulators, both operands along the sum; N / 8 from bit 17, M / 16 from bit 24
          const uint32_t shape = 1u << 4 | 1u << 7 | 1u << 10 | (uint32_t)(width / 8) << 17 | (uint32_t)(kM / 16) << 24;
          for (int left = now.chunks; left > 0; --left, ++j) {
            // steps of the descriptors' address field, 16 bytes each; it does not overflow
            const uint64_t da = a0 + (j & 1) * (operand_bytes(kM) >> 4), db = b0 + (j & 1) * (operand_bytes(kN) >> 4);
            const uint32_t d = tmem + (uint32_t)((j & 1) * kN);
            if (SPLIT_B) wait_for(arrived0, j);
            wait_for(filled0, j);
            if (!good) break;  // who waits for this chunk gives up too
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            constexpr int kPairs[6][2] = {{0, 2}, {2, 0}, {1, 1}, {0, 1}, {1, 0}, {0, 0}};
#pragma unroll
            for (int p = 0; p < 6; ++p)
#pragma unroll
              for (int k = 0; k < kChunk / 16; ++k) {
                const uint64_t pa = da + (kPairs[p][0] * kGroups + 2 * k) * (group_stride(kM) >> 4);
                const uint64_t qb = db + (kPairs[p][1] * kGroups + 2 * k) * (uint32_t)(strb >> 4);
                const bool scaled = p > 0 && k == 0 && kPairs[p][0] + kPairs[p][1] < kPairs[p - 1][0] + kPairs[p - 1][1];
                if (scaled) mma<kPartBits>(d, pa, qb, shape, true);
                else mma<0>(d, pa, qb, shape, p + k > 0);
              }
            asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                             done0 + 8 * (j & 1))
                         : "memory");
          }
        }
        if (!good) {  // the instructions in flight end before the tensor memory is given back
          asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                           smem_address(&idle))
                       : "memory");
          mbarrier_wait(smem_address(&idle), 0, smem_address(&never));
        }
      }
      __syncwarp();
    } else if (warp == kWarps + 1) {
      // ---- the image's copies, two chunks ahead; one lane works
      if (SPLIT_B && lane == 0) {
        int j = 0;
        for (int i = blockIdx.x; i < items && good; i += gridDim.x) {
          const Item now = item_of<kN>(a, i);
          const uint32_t bytes = operand_bytes(tile_width<kN>(a.rows_b, now.n0));
          const unsigned char* from = a.image + (int64_t)(now.n0 / kN) * now.chunks * operand_bytes(kN);
          for (int left = now.chunks; left > 0; --left, ++j, from += bytes) {
            if (j >= 2) wait_for(done0, j - 2);
            if (!good) break;
            bulk_copy(smem_address(smem + S::kB + (j & 1) * operand_bytes(kN)), from, bytes, arrived0 + 8 * (j & 1));
          }
        }
        // the copies in flight have arrived before the block ends; their readers wait for them otherwise
        for (int k = j > 2 ? j - 2 : 0; !good && k < j; ++k)
          mbarrier_wait(arrived0 + 8 * (k & 1), k >> 1 & 1, smem_address(&never));
      }
      __syncwarp();
    }
  }
  __syncthreads();
  if (warp < kWarps && expired) give_up<kN>(a);
  if (warp == kWarps)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem) : "memory");
}

// The parts of B in the order and layout of the stages: per tile of columns, per chunk.
template <bool ALONG>
__global__ void __launch_bounds__(256) split_kernel(const float* __restrict__ B, int64_t ld, int rows, int depth,
                                                    unsigned char* __restrict__ image) {
  constexpr int kN = Shape<true>::kN;
  const int chunks = (depth + kChunk - 1) / kChunk;
  const int n0 = blockIdx.y * kN, width = tile_width<kN>(rows, n0), stride = group_stride(width);
  const int i = blockIdx.x * 256 + threadIdx.x;  // (chunk, row, group), or (chunk, group, row)
  const int row = ALONG ? i / kGroups % width : i % width;
  const int group = ALONG ? i % kGroups : i / width % kGroups;
  const int chunk = i / (kGroups * width);
  if (chunk >= chunks) return;
  float x[8];
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const int k = chunk * kChunk + group * 8 + q;
    x[q] = n0 + row < rows && k < depth ? element<ALONG>(B, ld, n0 + row, k) : 0.f;
  }
  put(image + (int64_t)blockIdx.y * chunks * operand_bytes(kN) + (int64_t)chunk * operand_bytes(width) + group * stride +
          row * 16,
      stride, x);
}

// dW = the sum of the slices, always in the same order.  A warp's lanes read neighbouring elements.
__global__ void __launch_bounds__(256) sum_slices_kernel(const float* __restrict__ partial, int slices, int64_t count,
                                                         float* __restrict__ out) {
  const int64_t i = (int64_t)blockIdx.x * 256 + threadIdx.x;
  if (i >= count) return;
  float s[4] = {0.f, 0.f, 0.f, 0.f};
  int k = 0;
  for (; k + 4 <= slices; k += 4)
#pragma unroll
    for (int j = 0; j < 4; ++j) s[j] += partial[(int64_t)(k + j) * count + i];
  for (; k < slices; ++k) s[0] += partial[(int64_t)k * count + i];
  out[i] = (s[0] + s[1]) + (s[2] + s[3]);
}

// rows of whole units of `unit` floats, the first on a boundary
bool aligned_rows(const float* p, int64_t ld, int unit) {
  return ld % unit == 0 && reinterpret_cast<uintptr_t>(p) % (4 * unit) == 0;
}

template <bool ALONG_A, bool ALONG_B, bool SPLIT_B>
dg_status_t launch(const Graph* g, const LinearArgs& a, cudaStream_t s) {
  const int64_t items = (int64_t)a.tiles_m * a.tiles_n * a.slices;
  auto kernel = linear_kernel<ALONG_A, ALONG_B, SPLIT_B>;
  DG_CUDA(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               Shape<SPLIT_B>::kBytes));
  kernel<<<(unsigned)(items < g->sm_count ? items : g->sm_count), kThreads, Shape<SPLIT_B>::kBytes, s>>>(a);
  DG_CUDA(cudaGetLastError());
  count_launches(1);
  return DG_OK;
}

template <bool SPLIT_B>
void fill(LinearArgs* a) {
  a->tiles_m = (a->rows_a + kM - 1) / kM;
  a->tiles_n = (a->rows_b + Shape<SPLIT_B>::kN - 1) / Shape<SPLIT_B>::kN;
  a->vector_a = aligned_rows(a->A, a->lda, 4);
  a->vector_b = aligned_rows(a->B, a->ldb, 4);
  a->vector_out = aligned_rows(a->out, a->rows_b, 4);
  a->linear_out = !a->vector_out && a->rows_b <= 48 && a->slices == 1 && aligned_rows(a->out, 4, 4);
}

// A layer's product with its weights as B: split first, where there is memory for it.
template <bool ALONG_B>
dg_status_t with_weights(const Graph* g, LinearArgs a, cudaStream_t s) {
  fill<true>(&a);
  constexpr int kN = Shape<true>::kN;
  const int64_t chunks = (a.depth + kChunk - 1) / kChunk;
  void* image = nullptr;
  if (scratch_alloc(g, (size_t)a.tiles_n * (size_t)chunks * (size_t)operand_bytes(kN), s, &image) !=
      cudaSuccess) {
    fill<false>(&a);
    return launch<true, ALONG_B, false>(g, a, s);
  }
  const unsigned blocks = (unsigned)((chunks * kGroups * kN + 255) / 256);
  split_kernel<ALONG_B><<<dim3(blocks, (unsigned)a.tiles_n), 256, 0, s>>>(a.B, a.ldb, a.rows_b, a.depth,
                                                                         static_cast<unsigned char*>(image));
  dg_status_t st = DG_OK;
  if (const cudaError_t e = cudaGetLastError()) {
    st = cuda_fail(e, "splitting the weights");
  } else {
    count_launches(1);
    a.image = static_cast<const unsigned char*>(image);
    st = launch<true, ALONG_B, true>(g, a, s);
  }
  pool_free(image, s);
  return st;
}

}  // namespace

dg_status_t linear_expired(int64_t* blocks) {
  unsigned long long count = 0;
  DG_CUDA(cudaDeviceSynchronize());
  DG_CUDA(cudaMemcpyFromSymbol(&count, g_expired, sizeof(count)));
  *blocks = (int64_t)count;
  return DG_OK;
}

dg_status_t linear_fwd(const Graph* g, const float* X, int32_t K, const float* W, int32_t N, const float* scale,
                       const float* bias, bool relu, float* Y, cudaStream_t s) {
  LinearArgs a{};
  a.A = X;
  a.lda = K;
  a.rows_a = (int)g->n;
  a.B = W;
  a.ldb = K;
  a.rows_b = N;
  a.depth = a.depth_slice = K;
  a.slices = 1;
  a.scale = scale;
  a.bias = bias;
  a.relu = relu;
  a.out = Y;
  return with_weights<true>(g, a, s);
}

dg_status_t linear_bwd_input(const Graph* g, const float* G, int32_t N, const float* W, int32_t K, float* dX,
                             cudaStream_t s) {
  LinearArgs a{};
  a.A = G;
  a.lda = N;
  a.rows_a = (int)g->n;
  a.B = W;
  a.ldb = K;
  a.rows_b = K;
  a.depth = a.depth_slice = N;
  a.slices = 1;
  a.out = dX;
  return with_weights<false>(g, a, s);
}

dg_status_t linear_bwd_weight(const Graph* g, const float* G, int32_t N, const float* X, int32_t K, float* dW,
                              cudaStream_t s) {
  LinearArgs a{};
  a.A = G;
  a.lda = N;
  a.rows_a = N;
  a.B = X;
  a.ldb = K;
  a.rows_b = K;
  a.depth = (int)g->n;
  // as many slices as fill the SMs, of at least 16 chunks each
  const int64_t tiles = (int64_t)((N + kM - 1) / kM) * ((K + kM - 1) / kM);
  int64_t slices = g->sm_count / tiles;
  const int64_t most = (g->n + 16 * kChunk - 1) / (16 * kChunk);
  if (slices > most) slices = most;
  // Fewer where the scratch holds fewer, down to one, which takes no memory.  245 k rows of 256 x 256: 37 slices 269 us,
  // 20 481, 16 597, 8 1186, 4 2342, one 9317.
  const int64_t slice_bytes = (int64_t)N * K * (int64_t)sizeof(float);
  if (slices > (g->scratch_mb << 20) / slice_bytes) slices = (g->scratch_mb << 20) / slice_bytes;
  void* partial = nullptr;
  while (slices > 1 && scratch_alloc(g, (size_t)(slices * slice_bytes), s, &partial) != cudaSuccess) slices /= 2;
  if (slices < 1) slices = 1;
  int64_t slice = (g->n + slices - 1) / slices;
  slice = (slice + kChunk - 1) / kChunk * kChunk;
  a.depth_slice = (int)(slice < g->n ? slice : g->n);
  a.slices = (int)((g->n + a.depth_slice - 1) / a.depth_slice);
  a.out = partial ? static_cast<float*>(partial) : dW;
  fill<false>(&a);
  dg_status_t st = launch<false, false, false>(g, a, s);
  if (st == DG_OK && partial) {
    const int64_t count = (int64_t)N * K;
    sum_slices_kernel<<<(unsigned)((count + 255) / 256), 256, 0, s>>>(static_cast<float*>(partial), a.slices, count, dW);
    if (const cudaError_t e = cudaGetLastError()) st = cuda_fail(e, "sum of the slices");
    else count_launches(1);
  }
  pool_free(partial, s);
  return st;
}

}  // namespace dg
