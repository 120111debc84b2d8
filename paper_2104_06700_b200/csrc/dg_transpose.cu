// CSR -> CSC on the GPU as a stable least-significant-digit radix sort of (key = colidx[k],
// value = k).  The paper keeps the graph in CSR only (Section 3.1) and leaves the reverse graph
// of the backward pass implicit; the result here is defined as the stable counting sort of the
// edge positions by source vertex, which has exactly one correct answer.
//
// The digits are 8 bits wide, or 9 where that pays (see sort_plan).  One pass over a digit is
// three kernels and never makes one block wait for another:
//   1. digit_histogram : per tile of kTile keys, the number of keys per digit -> hist[digit][tile]
//   2. exclusive scan of hist (digit-major, so the scan yields global output offsets):
//      scan_reduce -> scan_spine (one block) -> scan_apply, or scan_few
//   3. digit_scatter   : ranks every key inside its tile in input order (ballots over the digit
//      bits inside a warp, per-warp counters across rounds, a fixed pass across the warps), stages
//      the tile sorted by digit in shared memory and writes each digit run to its global offset.
// Stability of every step makes the final order (key, k) ascending.
//
// The last pass of a transposition does not write the keys again: it counts the columns (the entries of a column lie
// side by side in a sorted tile), and writes beside perm the row of every entry, which it finds in a table of 16 bytes per
// 32 positions, and the row's factor.  That saves the passes that read the sorted keys, wrote (row, factor) pairs of 8 bytes
// per edge and gathered them through perm, one random DRAM read per edge; the table of 124 M edges is 62 MB and its reads
// hit L2.  Create and transposition, us before / after: 124 M edges, 2.4 M vertices 4670 / 3945; 81 M edges, 5.6 M vertices
// 3758 / 2825; 115 M edges, 233 k vertices 4540 / 4000; 576 M edges 37100 / 34500; 65 k edges 138 / 131.  Rows carried through
// the passes instead, with two passes of 11 bits or three of 8: 4150 and 4096.
#include "dg_internal.cuh"

namespace dg {
namespace {

constexpr int kMaxRadixBits = 9;
constexpr int kSortBlock = 256;
constexpr int kSortWarps = kSortBlock / 32;
constexpr int kItems = 16;                       // keys per thread
constexpr int kTile = kSortBlock * kItems;       // 4096 keys per block
constexpr int kScanBlock = 256;
constexpr int kScanItems = 16;
constexpr int kScanChunk = kScanBlock * kScanItems;
constexpr unsigned kFull = 0xffffffffu;

// The kernels of a sort follow one another closely (see launch_kernel): the next one's blocks come up while this one's last
// run, and wait here for its end.  A small graph's ingest is the gaps between launches (create and transposition of 1.2 M
// edges 179 -> 156 us, of 31 M 1308 -> 1277).
__device__ __forceinline__ void overlap_begin() {
  cudaGridDependencySynchronize();
  cudaTriggerProgrammaticLaunchCompletion();
}

template <int BITS>
__device__ __forceinline__ uint32_t digit_of(uint32_t key, int shift) {
  return (key >> shift) & ((1u << BITS) - 1u);
}

// A thread reads its keys as 16-byte vectors when the array allows it (four loads in flight
// then cover the whole tile; with 4-byte loads the kernel waited on memory at a third of the
// copy bandwidth).  The caller's colidx, the keys of the first pass, is only 4-byte aligned in
// general: `vector_ok` says whether keys is 16-byte aligned.
template <int BITS>
__global__ void __launch_bounds__(kSortBlock)
digit_histogram(const uint32_t* __restrict__ keys, int64_t count, int shift, int64_t tiles,
                int vector_ok, uint32_t* __restrict__ hist) {
  overlap_begin();
  constexpr int R = 1 << BITS;
  __shared__ uint32_t h[R];
  for (int d = threadIdx.x; d < R; d += kSortBlock) h[d] = 0;
  __syncthreads();
  const int64_t base = (int64_t)blockIdx.x * kTile;
  if (vector_ok && base + kTile <= count) {
    const uint4* v = reinterpret_cast<const uint4*>(keys + base);
    uint4 k[kItems / 4];
#pragma unroll
    for (int i = 0; i < kItems / 4; ++i) k[i] = v[i * kSortBlock + threadIdx.x];
#pragma unroll
    for (int i = 0; i < kItems / 4; ++i) {
      atomicAdd(&h[digit_of<BITS>(k[i].x, shift)], 1u);
      atomicAdd(&h[digit_of<BITS>(k[i].y, shift)], 1u);
      atomicAdd(&h[digit_of<BITS>(k[i].z, shift)], 1u);
      atomicAdd(&h[digit_of<BITS>(k[i].w, shift)], 1u);
    }
  } else {
#pragma unroll 4
    for (int i = 0; i < kItems; ++i) {
      const int64_t k = base + i * kSortBlock + threadIdx.x;
      if (k < count) atomicAdd(&h[digit_of<BITS>(keys[k], shift)], 1u);
    }
  }
  __syncthreads();
  for (int d = threadIdx.x; d < R; d += kSortBlock) hist[(int64_t)d * tiles + blockIdx.x] = h[d];
}

// ---- exclusive scan of a uint32 array of length m (in place), three kernels ----
template <int THREADS>
__device__ __forceinline__ uint32_t block_exclusive_scan(uint32_t v, uint32_t* total) {
  __shared__ uint32_t warp_sums[THREADS / 32];
  __shared__ uint32_t block_total;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint32_t inc = v;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const uint32_t t = __shfl_up_sync(kFull, inc, d);
    if (lane >= d) inc += t;
  }
  if (lane == 31) warp_sums[warp] = inc;
  __syncthreads();
  if (warp == 0) {
    uint32_t w = lane < THREADS / 32 ? warp_sums[lane] : 0;
    uint32_t winc = w;
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
      const uint32_t t = __shfl_up_sync(kFull, winc, d);
      if (lane >= d) winc += t;
    }
    if (lane < THREADS / 32) warp_sums[lane] = winc - w;
    if (lane == THREADS / 32 - 1) block_total = winc;
  }
  __syncthreads();
  const uint32_t r = inc - v + warp_sums[warp];
  *total = block_total;
  __syncthreads();  // the shared arrays may be reused by the next call
  return r;
}

__global__ void __launch_bounds__(kScanBlock)
scan_reduce(const uint32_t* __restrict__ data, int64_t m, uint32_t* __restrict__ chunk_sums) {
  overlap_begin();
  const int64_t base = (int64_t)blockIdx.x * kScanChunk + (int64_t)threadIdx.x * kScanItems;
  uint32_t s = 0;
#pragma unroll
  for (int i = 0; i < kScanItems; ++i)
    if (base + i < m) s += data[base + i];
  uint32_t total;
  block_exclusive_scan<kScanBlock>(s, &total);
  if (threadIdx.x == 0) chunk_sums[blockIdx.x] = total;
}

// `stride` words from one chunk's sum to the next
__global__ void __launch_bounds__(kScanBlock)
scan_spine(uint32_t* __restrict__ chunk_sums, int64_t stride, int64_t chunks) {
  overlap_begin();
  uint32_t carry = 0;
  for (int64_t base = 0; base < chunks; base += kScanBlock) {
    const int64_t i = base + threadIdx.x;
    const uint32_t v = i < chunks ? chunk_sums[i * stride] : 0;
    uint32_t total;
    const uint32_t ex = block_exclusive_scan<kScanBlock>(v, &total);
    if (i < chunks) chunk_sums[i * stride] = carry + ex;
    carry += total;
  }
}

__global__ void __launch_bounds__(kScanBlock)
scan_apply(uint32_t* __restrict__ data, int64_t m, const uint32_t* __restrict__ chunk_sums) {
  overlap_begin();
  const int64_t base = (int64_t)blockIdx.x * kScanChunk + (int64_t)threadIdx.x * kScanItems;
  uint32_t v[kScanItems];
  uint32_t s = 0;
#pragma unroll
  for (int i = 0; i < kScanItems; ++i) {
    v[i] = base + i < m ? data[base + i] : 0;
    s += v[i];
  }
  uint32_t total;
  uint32_t run = block_exclusive_scan<kScanBlock>(s, &total) + chunk_sums[blockIdx.x];
#pragma unroll
  for (int i = 0; i < kScanItems; ++i) {
    if (base + i < m) data[base + i] = run;
    run += v[i];
  }
}

// The whole scan in one block: of up to kFewEntries, one launch instead of three (a second round of the block takes ten
// microseconds).  PAIRS: `data` are the pairs below, and 64-bit sums take their place.
constexpr int kFewThreads = 1024;
constexpr int64_t kFewEntries = kFewThreads * kScanItems;
template <bool PAIRS>
__global__ void __launch_bounds__(kFewThreads) scan_few(uint32_t* __restrict__ data, int64_t m) {
  overlap_begin();
  const int base = threadIdx.x * kScanItems;
  uint32_t v[kScanItems], s = 0;
  // whole shares by 16 bytes: number by number a warp's loads spread over 64 lines each (15.6 k entries: transposition of
  // 247 k edges 99 us, so 77, and 86 with three launches)
  const bool whole = base + kScanItems <= m;
  if (whole) {
#pragma unroll
    for (int i = 0; i < kScanItems; i += PAIRS ? 2 : 4) {
      const uint4 q = *reinterpret_cast<const uint4*>(data + (PAIRS ? 2 * (base + i) : base + i));
      v[i] = q.x;
      if (PAIRS) {
        v[i + 1] = q.z;
      } else {
        v[i + 1] = q.y; v[i + 2] = q.z; v[i + 3] = q.w;
      }
    }
  } else {
#pragma unroll
    for (int i = 0; i < kScanItems; ++i) v[i] = base + i < m ? data[PAIRS ? 2 * (base + i) : base + i] : 0u;
  }
#pragma unroll
  for (int i = 0; i < kScanItems; ++i) s += v[i];
  uint32_t total;
  uint32_t run = block_exclusive_scan<kFewThreads>(s, &total);
  if (whole) {
#pragma unroll
    for (int i = 0; i < kScanItems; i += PAIRS ? 2 : 4) {
      uint4 q;
      if (PAIRS) {
        q = make_uint4(run, 0u, run + v[i], 0u);
        run = q.z + v[i + 1];
      } else {
        q.x = run; q.y = q.x + v[i]; q.z = q.y + v[i + 1]; q.w = q.z + v[i + 2];
        run = q.w + v[i + 3];
      }
      *reinterpret_cast<uint4*>(data + (PAIRS ? 2 * (base + i) : base + i)) = q;
    }
    return;
  }
#pragma unroll
  for (int i = 0; i < kScanItems; ++i) {
    if (base + i < m) {
      if (PAIRS) reinterpret_cast<int64_t*>(data)[base + i] = (int64_t)run;
      else data[base + i] = run;
    }
    run += v[i];
  }
}

// ---- the column pointers, from counts ----
// While the edges are sorted, colptr holds a pair per column: x the entries counted so far, y the bits of the factor
// 1/(in-degree + self) of the vertex.  Then it is scanned in place; the sum of a chunk of kScanChunk columns travels
// in y of the chunk's first pair.
__global__ void __launch_bounds__(256)
columns_begin_kernel(const int64_t* __restrict__ rowptr, int64_t n, int self, uint2* __restrict__ columns) {
  overlap_begin();
  const int64_t v = (int64_t)blockIdx.x * 256 + threadIdx.x;
  if (v > n) return;
  float inv = 0.f;
  if (v < n) inv = 1.0f / (float)(__ldg(rowptr + v + 1) - __ldg(rowptr + v) + self);
  columns[v] = make_uint2(0u, __float_as_uint(inv));
}

__global__ void __launch_bounds__(kScanBlock)
columns_reduce(uint2* __restrict__ columns, int64_t m) {
  overlap_begin();
  const int64_t chunk = (int64_t)blockIdx.x * kScanChunk;
  uint32_t s = 0;
#pragma unroll
  for (int i = 0; i < kScanItems; ++i) {
    const int64_t u = chunk + i * kScanBlock + threadIdx.x;
    if (u < m) s += columns[u].x;
  }
  uint32_t total;
  block_exclusive_scan<kScanBlock>(s, &total);
  if (threadIdx.x == 0) columns[chunk].y = total;
}

__global__ void __launch_bounds__(kScanBlock)
columns_apply(uint2* __restrict__ columns, int64_t m) {
  overlap_begin();
  const int64_t chunk = (int64_t)blockIdx.x * kScanChunk, base = chunk + (int64_t)threadIdx.x * kScanItems;
  const uint32_t before = columns[chunk].y;  // read by all before the barriers below let anyone write it
  uint32_t v[kScanItems], s = 0;
#pragma unroll
  for (int i = 0; i < kScanItems; ++i) {
    v[i] = base + i < m ? columns[base + i].x : 0u;
    s += v[i];
  }
  uint32_t total;
  uint32_t run = before + block_exclusive_scan<kScanBlock>(s, &total);
#pragma unroll
  for (int i = 0; i < kScanItems; ++i) {
    if (base + i < m) reinterpret_cast<int64_t*>(columns)[base + i] = (int64_t)run;
    run += v[i];
  }
}

// ---- the row of a position ----
// table[b] for the positions 32 b ... 32 b + 31: x the row r of the first; y a bit for every other position that begins a
// row, so that the row of position 32 b + i is r + the number of bits 1 ... i; bit 0: a row without entries lies between
// them, and the count is wrong; z, w: the bits of the factors of r and r + 1, where most entries belong (one random
// read instead of two).
struct RowOf {
  int64_t row;
  bool known;       // `factor` is the row's
  uint32_t factor;
};
__device__ __forceinline__ RowOf row_of(const uint4* __restrict__ table, const int64_t* __restrict__ rowptr, int64_t n,
                                        int64_t nnz, uint32_t k, const uint4& block) {
  if (!(block.y & 1u)) {
    const int later = __popc(block.y & ((2u << (k & 31u)) - 1u));
    return {(int64_t)block.x + later, later < 2, later ? block.w : block.z};
  }
  const int64_t b = (int64_t)(k >> 5) + 1;
  int64_t lo = block.x, hi = 32 * b < nnz ? (int64_t)__ldg(&table[b].x) + 1 : n;  // the last row that begins at or before k
  while (hi - lo > 1) {
    const int64_t mid = (lo + hi) >> 1;
    if (__ldg(rowptr + mid) <= (int64_t)k) lo = mid;
    else hi = mid;
  }
  return {lo, false, 0u};
}

// A warp takes one chunk of the rows' plan (see Plan).  The bits are zero before.
__global__ void __launch_bounds__(256)
row_table_kernel(const Chunk* __restrict__ chunks, int32_t chunk_count, const int64_t* __restrict__ rowptr, int64_t n,
                 const uint2* __restrict__ columns, uint4* __restrict__ table) {
  overlap_begin();
  const int lane = threadIdx.x & 31;
  const int chunk = blockIdx.x * 8 + __shfl_sync(kFull, (int)(threadIdx.x >> 5), 0);
  if (chunk >= chunk_count) return;
  const int4 here = __ldg(reinterpret_cast<const int4*>(chunks) + chunk);
  const int4 next = __ldg(reinterpret_cast<const int4*>(chunks) + chunk + 1);
  const int nrows = here.z >= 0 ? 1 : next.x - here.x + (next.z >= 0 ? 1 : 0);
  Position begin = 0, end = 0;
  uint32_t factor = 0, following = 0;
  if (lane < nrows) {
    const int64_t r = here.x + lane;
    const int64_t row_begin = __ldg(rowptr + r), row_end = __ldg(rowptr + r + 1);
    begin = max((int)row_begin, here.y);
    end = min((int)row_end, next.y);
    factor = __ldg(&columns[r].y);
    following = r + 1 < n ? __ldg(&columns[r + 1].y) : 0u;
    if (row_begin < row_end && here.z < 0 && (row_begin & 31)) {  // a piece of a cut row begins no row
      const bool after_empty = r > 0 && __ldg(rowptr + r - 1) == row_begin;
      atomicOr(&table[row_begin >> 5].y, 1u << (row_begin & 31) | (after_empty ? 1u : 0u));
    }
  }
  for (int i = 0; i < nrows; ++i) {
    const Position lo = __shfl_sync(kFull, begin, i), hi = __shfl_sync(kFull, end, i);
    const uint2 factors = make_uint2(__shfl_sync(kFull, factor, i), __shfl_sync(kFull, following, i));
    for (Position b = ((lo + 31) >> 5) + lane; 32 * b < hi; b += 32) {
      table[b].x = (uint32_t)(here.x + i);
      *reinterpret_cast<uint2*>(&table[b].z) = factors;
    }
  }
}

// Lanes of the warp that hold the same digit as this lane (lanes without a key only match one
// another): one ballot per digit bit, each keeping the lanes that agree with this lane on that
// bit.  Unlike match.any, whose cost grows with the number of distinct values in the warp (about
// 30 for the random low digits of vertex ids), this costs the same for every digit mix.
template <int BITS>
__device__ __forceinline__ unsigned digit_peers(uint32_t d, bool valid) {
  const unsigned have = __ballot_sync(kFull, valid);
  unsigned peers = valid ? have : ~have;
#pragma unroll
  for (int b = 0; b < BITS; ++b) {
    const bool bit = (d >> b) & 1u;
    const unsigned m = __ballot_sync(kFull, bit);
    peers &= bit ? m : ~m;
  }
  return peers;
}

// ---- stable scatter of one tile ----
// vals_in == nullptr means "the value of key k is k" (first pass).
// The tile is staged in shared memory sorted by digit, one array after the other in the same 16 KB.
// Four blocks per SM (64 registers a thread): the ranking is a chain of shared-memory and ballot latencies.
// Values are read only when the keys have left their registers, and two places share one: nothing spills
// (0.78 -> 0.68 ms per pass over 124 M pairs; three blocks at 80 registers 1.02, five at 48 0.73).
// With CSC the last pass of a transposition: twice the time of a plain pass (18.6 M edges 258 us, a plain one 111), for
// the random reads of the table, four in flight per thread, and three arrays written instead of two.
struct CscArgs {  // empty otherwise
  const uint4* table;     // see row_of
  const int64_t* rowptr;
  int64_t n;
  uint2* columns;         // see columns_begin_kernel
  int32_t* rows_out;
  float* scale_out;       // the factor of every entry's row
};
template <int BITS, bool CSC>
__global__ void __launch_bounds__(kSortBlock, 4)
digit_scatter(const uint32_t* __restrict__ keys_in, const uint32_t* __restrict__ vals_in,
              int64_t count, int shift, int64_t tiles, const uint32_t* __restrict__ offsets,
              uint32_t* __restrict__ keys_out, uint32_t* __restrict__ vals_out, const CscArgs c) {
  overlap_begin();
  constexpr int R = 1 << BITS;
  constexpr int DPT = R / kSortBlock;  // digits a thread owns (consecutive ones): 1 or 2
  // A warp ranks its 512 keys as two streams of 256 (rounds 0..7 and 8..15), each with its own
  // counters, so that two independent chains of counter updates are in flight at a time.
  // Dynamic shared memory (36 KB with 9-bit digits): cnt_a, cnt_b, digit_base, global_base, stage.
  extern __shared__ __align__(16) unsigned char scatter_smem[];
  uint16_t (*cnt_a)[R] = reinterpret_cast<uint16_t (*)[R]>(scatter_smem);
  uint16_t (*cnt_b)[R] = cnt_a + kSortWarps;
  uint32_t* digit_base = reinterpret_cast<uint32_t*>(cnt_b + kSortWarps);
  uint32_t* global_base = digit_base + R;
  uint32_t* stage = global_base + R;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const unsigned lt_mask = (1u << lane) - 1u;
  const int64_t tile_base = (int64_t)blockIdx.x * kTile;
  const int64_t remaining = count - tile_base;
  const int tile_count = remaining < kTile ? (int)remaining : kTile;

  // this tile's global offsets of the thread's digits: fetched now, needed after the ranking
  uint32_t my_global_base[DPT];
#pragma unroll
  for (int i = 0; i < DPT; ++i)
    my_global_base[i] = offsets[(int64_t)(threadIdx.x * DPT + i) * tiles + blockIdx.x];
  for (int w = 0; w < kSortWarps; ++w) {
#pragma unroll
    for (int i = 0; i < DPT; ++i) {
      cnt_a[w][threadIdx.x * DPT + i] = 0;
      cnt_b[w][threadIdx.x * DPT + i] = 0;
    }
  }
  __syncthreads();

  // Warp `warp` owns keys [warp*512, warp*512+512) of the tile, 32 consecutive keys per round,
  // so (warp, round, lane) order is input order.
  uint32_t key[kItems];
  constexpr int kHalf = kItems / 2;
  uint32_t place[kHalf] = {};  // rank, later the place in the sorted tile: of key r low, of key r + kHalf high
  auto place_of = [&](int r) { return r < kHalf ? place[r] & 0xffffu : place[r - kHalf] >> 16; };
#pragma unroll
  for (int r = 0; r < kItems; ++r) {
    const int local = warp * (32 * kItems) + r * 32 + lane;
    key[r] = local < tile_count ? keys_in[tile_base + local] : 0u;
  }
#pragma unroll
  for (int r = 0; r < kHalf; ++r) {
#pragma unroll
    for (int stream = 0; stream < 2; ++stream) {
      const int rr = r + stream * kHalf;
      uint16_t* cnt = stream ? cnt_b[warp] : cnt_a[warp];
      const bool valid = warp * (32 * kItems) + rr * 32 + lane < tile_count;
      const uint32_t d = valid ? digit_of<BITS>(key[rr], shift) : 0u;
      const unsigned peers = digit_peers<BITS>(d, valid);
      const int leader = __ffs(peers) - 1;
      uint32_t before = 0;
      if (valid && lane == leader) {
        before = cnt[d];
        cnt[d] = (uint16_t)(before + __popc(peers));
      }
      before = __shfl_sync(kFull, before, leader);
      const uint32_t rank = before + __popc(peers & lt_mask);
      place[r] = stream ? place[r] | rank << 16 : rank;
    }
    __syncwarp();
  }
  __syncthreads();

  // a thread owns DPT consecutive digits: exclusive prefix over (warp, stream) inside each, then
  // over the digits
  {
    uint32_t in_digit[DPT];
    uint32_t mine = 0;
#pragma unroll
    for (int i = 0; i < DPT; ++i) {
      const int d = threadIdx.x * DPT + i;
      uint32_t run = 0;
#pragma unroll
      for (int w = 0; w < kSortWarps; ++w) {
        const uint32_t ca = cnt_a[w][d];
        cnt_a[w][d] = (uint16_t)run;
        run += ca;
        const uint32_t cb = cnt_b[w][d];
        cnt_b[w][d] = (uint16_t)run;
        run += cb;
      }
      in_digit[i] = run;
      mine += run;
    }
    uint32_t total;
    uint32_t start = block_exclusive_scan<kSortBlock>(mine, &total);
#pragma unroll
    for (int i = 0; i < DPT; ++i) {
      digit_base[threadIdx.x * DPT + i] = start;
      global_base[threadIdx.x * DPT + i] = my_global_base[i];
      start += in_digit[i];
    }
  }
  __syncthreads();

#pragma unroll
  for (int r = 0; r < kItems; ++r) {
    const int local = warp * (32 * kItems) + r * 32 + lane;
    if (local < tile_count) {
      const uint32_t d = digit_of<BITS>(key[r], shift);
      const uint32_t add = digit_base[d] + (r < kHalf ? cnt_a[warp][d] : cnt_b[warp][d]);
      place[r % kHalf] += r < kHalf ? add : add << 16;  // places are below 4096: no carry into the high half
      stage[place_of(r)] = key[r];
      // the key has been staged: its register takes the value, on its way while the keys are written
      key[r] = vals_in ? vals_in[tile_base + local] : (uint32_t)(tile_base + local);
    }
  }
  __syncthreads();
  uint32_t dst[kItems];
#pragma unroll
  for (int j = 0; j < kItems; ++j) {
    const int i = j * kSortBlock + threadIdx.x;
    if (i < tile_count) {
      const uint32_t k = stage[i];
      const uint32_t d = digit_of<BITS>(k, shift);
      dst[j] = global_base[d] + ((uint32_t)i - digit_base[d]);
      if (!CSC) {
        keys_out[dst[j]] = k;
      } else if (k < (uint32_t)c.n) {  // an id outside the graph must not turn into a write outside the pairs
        // a column's entries of this tile lie side by side: the two ends of the run make the count
        if (i == 0 || stage[i - 1] != k) atomicAdd(&c.columns[k].x, 0u - (uint32_t)i);
        if (i == tile_count - 1 || stage[i + 1] != k) atomicAdd(&c.columns[k].x, (uint32_t)i + 1u);
      }
    }
  }
  __syncthreads();
#pragma unroll
  for (int r = 0; r < kItems; ++r) {
    const int local = warp * (32 * kItems) + r * 32 + lane;
    if (local < tile_count) {
      stage[place_of(r)] = key[r];
    }
  }
  __syncthreads();
  if (!CSC) {
#pragma unroll
    for (int j = 0; j < kItems; ++j) {
      const int i = j * kSortBlock + threadIdx.x;
      if (i < tile_count) vals_out[dst[j]] = stage[i];
    }
    return;
  }
  constexpr int kAhead = 4;  // look-ups in flight
#pragma unroll
  for (int j0 = 0; j0 < kItems; j0 += kAhead) {
    uint4 block[kAhead];
#pragma unroll
    for (int j = 0; j < kAhead; ++j) {
      const int i = (j0 + j) * kSortBlock + threadIdx.x;
      if (i < tile_count) block[j] = __ldg(c.table + (stage[i] >> 5));
    }
#pragma unroll
    for (int j = 0; j < kAhead; ++j) {
      const int i = (j0 + j) * kSortBlock + threadIdx.x;
      if (i < tile_count) {
        const uint32_t k = stage[i];
        const RowOf at = row_of(c.table, c.rowptr, c.n, count, k, block[j]);
        vals_out[dst[j0 + j]] = k;
        c.rows_out[dst[j0 + j]] = (int32_t)at.row;
        c.scale_out[dst[j0 + j]] = __uint_as_float(at.known ? at.factor : __ldcg(&c.columns[at.row].y));
      }
    }
  }
}

template <int BITS>
constexpr size_t scatter_smem_bytes() {
  return (size_t)2 * kSortWarps * (1 << BITS) * sizeof(uint16_t) + (size_t)2 * (1 << BITS) * sizeof(uint32_t) +
         (size_t)kTile * sizeof(uint32_t);
}

// colptr[u] = first position q whose sorted key is >= u.  Position q fills the ids between the
// key before it and its own key; position nnz closes the array up to n.  A thread takes
// kColptrItems consecutive positions (16-byte loads when `vector_ok`: sorted 16-byte aligned)
// and fills at most the last kMaxFill ids of a gap itself: a long run of ids without a key (a
// hub-first numbering puts every vertex without out-edges at the end, millions of them) would
// otherwise be one thread's loop (Papers-like x0.1, hub-first: 17 ms).  The ids it leaves keep
// the -1 the array was filled with, and fill_long_gaps finds each by a binary search.
// Eight positions and a shuffle for the key before them, instead of four and a load: 253 -> 213 us for 124 M keys.
constexpr int kColptrItems = 8;
constexpr int kMaxFill = 32;
__global__ void colptr_from_sorted_keys(const uint32_t* __restrict__ sorted, int64_t nnz,
                                        int64_t n, int vector_ok, int64_t* __restrict__ colptr) {
  const int64_t q0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) * kColptrItems;
  uint32_t k[kColptrItems];
  if (vector_ok && q0 + kColptrItems <= nnz) {
#pragma unroll
    for (int i = 0; i < kColptrItems; i += 4) {
      const uint4 v = *reinterpret_cast<const uint4*>(sorted + q0 + i);
      k[i] = v.x; k[i + 1] = v.y; k[i + 2] = v.z; k[i + 3] = v.w;
    }
  } else {
#pragma unroll
    for (int i = 0; i < kColptrItems; ++i) k[i] = q0 + i < nnz ? sorted[q0 + i] : 0u;
  }
  const uint32_t before = __shfl_up_sync(kFull, k[kColptrItems - 1], 1);
  if (q0 > nnz) return;
  int64_t prev = -1;
  if (q0 > 0) prev = (threadIdx.x & 31) ? before : sorted[q0 - 1];
#pragma unroll
  for (int i = 0; i < kColptrItems; ++i) {
    const int64_t q = q0 + i;
    if (q > nnz) break;
    int64_t cur = q < nnz ? (int64_t)k[i] : n;
    const int64_t next_prev = cur;
    if (cur > n) cur = n;  // an id outside [0, n) must not turn into a write outside colptr
    if (cur > prev) {
      int64_t u = prev + 1;
      if (cur - u >= kMaxFill) u = cur - kMaxFill + 1;
      for (; u <= cur; ++u) colptr[u] = q;
    }
    prev = next_prev;
  }
}

// the ids colptr_from_sorted_keys left at -1: the first position whose key is >= u, by search
__global__ void fill_long_gaps(const uint32_t* __restrict__ sorted, int64_t nnz, int64_t n,
                               int64_t* __restrict__ colptr) {
  const int64_t u = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (u > n || colptr[u] >= 0) return;
  int64_t lo = 0, hi = nnz;  // invariant: keys before lo are < u, keys from hi on are >= u
  while (lo < hi) {
    const int64_t mid = (lo + hi) >> 1;
    if ((int64_t)__ldg(sorted + mid) < u) lo = mid + 1;
    else hi = mid;
  }
  colptr[u] = lo;
}

constexpr int kRowItems = 8;
// out[k] = map[r] (or r) for the row r that holds position k.  A thread takes kRowItems consecutive
// positions: one binary search for the first, then a galloping search forward from the previous row for
// each of the others (rows are usually a few positions long, empty rows are skipped in doubling strides).
__global__ void expand_rows_kernel(const int64_t* __restrict__ rowptr, int64_t n, int64_t nnz,
                                   const int32_t* __restrict__ map, uint32_t* __restrict__ out) {
  const int64_t k0 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) * kRowItems;
  if (k0 >= nnz) return;
  int64_t lo = 0, hi = n;  // invariant: rowptr[lo] <= k0 < rowptr[hi]
  while (hi - lo > 1) {
    const int64_t mid = (lo + hi) >> 1;
    if (__ldg(rowptr + mid) <= k0) lo = mid; else hi = mid;
  }
  int64_t r = lo;
  int64_t r_end = __ldg(rowptr + r + 1);
  uint32_t payload = map ? (uint32_t)__ldg(map + r) : (uint32_t)r;
#pragma unroll 1
  for (int i = 0; i < kRowItems; ++i) {
    const int64_t k = k0 + i;
    if (k >= nnz) break;
    if (k >= r_end) {
      int64_t step = 1, lo2 = r, hi2 = r + 1;
      while (hi2 < n && __ldg(rowptr + hi2) <= k) {
        lo2 = hi2;
        step <<= 1;
        hi2 = hi2 + step < n ? hi2 + step : n;
      }
      while (hi2 - lo2 > 1) {
        const int64_t mid = (lo2 + hi2) >> 1;
        if (__ldg(rowptr + mid) <= k) lo2 = mid; else hi2 = mid;
      }
      r = lo2;
      r_end = __ldg(rowptr + r + 1);
      payload = map ? (uint32_t)__ldg(map + r) : (uint32_t)r;
    }
    out[k] = payload;
  }
}

// The weight arrays of the CSC, from perm: the last step of a transposition, whose last pass has written the factors
// (TABULATED), and again after the caller changed edge_w in place (learnable edge weights), when mean_scale_T holds
// products and the in-degree comes from the CSR row pointer.  A thread takes four edges: their random reads are in
// flight together.  Transposition of weighted graphs, us, degrees from the row pointers / tabulated: 11.5 M edges 499 / 460,
// 39.6 M 1490 / 1345, 79 M 3083 / 2893, 124 M 5226 / 5157.  Weights read in the last sort pass instead, whose few warps wait
// for them: 39.6 M 1790, 79 M 3829.
template <bool TABULATED>
__global__ void __launch_bounds__(256)
gather_weights_kernel(const uint32_t* __restrict__ perm, int64_t nnz, const float* __restrict__ edge_w,
                      const int32_t* __restrict__ rowidx_T, const int64_t* __restrict__ rowptr, int self,
                      float* __restrict__ w_T, float* __restrict__ mean_scale_T) {
  overlap_begin();
  const int64_t q0 = ((int64_t)blockIdx.x * 256 + threadIdx.x) * 4;
  if (q0 >= nnz) return;
  if (nnz - q0 >= 4) {  // the arrays of the CSC are 256-byte aligned
    const uint4 k = *reinterpret_cast<const uint4*>(perm + q0);
    const float w[4] = {__ldg(edge_w + k.x), __ldg(edge_w + k.y), __ldg(edge_w + k.z), __ldg(edge_w + k.w)};
    float t[4];
    if (TABULATED) {
      const float4 f = *reinterpret_cast<const float4*>(mean_scale_T + q0);
      t[0] = w[0] * f.x; t[1] = w[1] * f.y; t[2] = w[2] * f.z; t[3] = w[3] * f.w;
    } else {
      const int4 v = *reinterpret_cast<const int4*>(rowidx_T + q0);
      const int32_t r[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
      for (int i = 0; i < 4; ++i)
        t[i] = w[i] * (1.0f / (float)(__ldg(rowptr + r[i] + 1) - __ldg(rowptr + r[i]) + self));
    }
    *reinterpret_cast<float4*>(w_T + q0) = make_float4(w[0], w[1], w[2], w[3]);
    *reinterpret_cast<float4*>(mean_scale_T + q0) = make_float4(t[0], t[1], t[2], t[3]);
    return;
  }
  for (int64_t q = q0; q < nnz; ++q) {
    const float w = edge_w[perm[q]];
    const int64_t v = rowidx_T[q];
    w_T[q] = w;
    mean_scale_T[q] =
        w * (TABULATED ? mean_scale_T[q] : 1.0f / (float)(__ldg(rowptr + v + 1) - __ldg(rowptr + v) + self));
  }
}

inline size_t align256(size_t x) { return (x + 255) & ~(size_t)255; }
inline int aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; }

struct Layout {
  // csc storage
  size_t colptr_off, rowidx_off, perm_off, w_off, mscale_off, split_off, csc_bytes;
  // scratch
  size_t keys_a_off, keys_b_off, vals_off, hist_off, sums_off, scratch_bytes;
  int64_t tiles, hist_len, chunks;
  int passes;
};

Layout make_layout(int64_t n, int64_t nnz, bool weighted) {
  Layout L{};
  size_t o = 0;
  L.colptr_off = o; o += align256((size_t)(n + 1) * 8);
  L.rowidx_off = o; o += align256((size_t)nnz * 4);
  L.perm_off = o;   o += align256((size_t)nnz * 4);
  L.w_off = o;      o += weighted ? align256((size_t)nnz * 4) : 0;
  L.mscale_off = o; o += align256((size_t)nnz * 4);
  L.split_off = o;  o += wants_split(n, nnz) ? align256((size_t)(kFineBlocks + 1) * n * 4) : 0;
  L.csc_bytes = o > 0 ? o : 256;
  L.passes = sort_plan(n).passes;
  L.tiles = (nnz + kTile - 1) / kTile;
  L.hist_len = L.tiles * (1 << kMaxRadixBits);
  L.chunks = (L.hist_len + kScanChunk - 1) / kScanChunk;
  o = 0;
  L.keys_a_off = o; o += align256((size_t)nnz * 4);
  L.keys_b_off = o; o += align256((size_t)nnz * 4);
  L.vals_off = o;   o += align256((size_t)nnz * 4);
  L.hist_off = o;   o += align256((size_t)L.hist_len * 4);
  L.sums_off = o;   o += align256((size_t)(L.chunks > 0 ? L.chunks : 1) * 4);
  L.scratch_bytes = o > 0 ? o : 256;
  return L;
}

}  // namespace

// Digit width and number of passes for keys in [0, key_range).  A 9-bit pass costs about a third
// more than an 8-bit one (nine ballots per ranking round, twice the counters and histogram, more
// spilled registers: measured on the 1.6 G-edge graph, 27 key bits, 3 x 9 bits took 100.3 ms
// against 98.1 ms for 4 x 8), so the wider digit is taken only where it turns three passes into
// two or two into one (key ranges of 9, 17 and 18 bits: the Reddit- and Proteins-like graphs,
// whose transposition gains 5 %).
SortPlan sort_plan(int64_t key_range) {
  int bits = 1;
  while (bits < 31 && ((int64_t)1 << bits) < key_range) ++bits;
  const int p8 = (bits + 7) / 8, p9 = (bits + 8) / 9;
  SortPlan plan;
  const bool wide = 4 * p9 < 3 * p8;
  plan.digit_bits = wide ? 9 : 8;
  plan.passes = wide ? p9 : p8;
  return plan;
}

// Sized for the wider digit, so that one workspace query serves every key range.
void sort_scratch_sizes(int64_t count, size_t* hist_bytes, size_t* sums_bytes) {
  const int64_t tiles = (count + kTile - 1) / kTile;
  const int64_t hist_len = tiles * (1 << kMaxRadixBits);
  const int64_t chunks = (hist_len + kScanChunk - 1) / kScanChunk;
  *hist_bytes = align256((size_t)(hist_len > 0 ? hist_len : 1) * 4);
  *sums_bytes = align256((size_t)(chunks > 0 ? chunks : 1) * 4);
}

template <int BITS>
static dg_status_t sort_passes_run(const uint32_t* keys_in, const uint32_t* vals_in, int64_t count,
                                   int passes, uint32_t* const keys_buf[2], uint32_t* vals_final,
                                   uint32_t* vals_tmp, uint32_t* hist,
                                   uint32_t* sums, const uint32_t** sorted_keys, CscArgs* csc,
                                   const Graph* g, cudaStream_t s) {
  const int64_t tiles = (count + kTile - 1) / kTile;
  const int64_t hist_len = tiles * (1 << BITS);
  const int64_t chunks = (hist_len + kScanChunk - 1) / kScanChunk;
  constexpr size_t smem = scatter_smem_bytes<BITS>();
  for (int p = 0; p < passes; ++p) {
    const int shift = p * BITS;
    // value buffers alternate so that the last pass lands in vals_final
    uint32_t* vals_out = ((passes - 1 - p) % 2 == 0) ? vals_final : vals_tmp;
    uint32_t* keys_out = keys_buf[p % 2];
    DG_CUDA(launch_kernel(digit_histogram<BITS>, dim3((unsigned)tiles), kSortBlock, s, true, keys_in, count, shift, tiles,
                          aligned16(keys_in), hist));
    if (hist_len <= kFewEntries) {
      DG_CUDA(launch_kernel(scan_few<false>, dim3(1), kFewThreads, s, true, hist, hist_len));
      count_launches(1);
    } else {
      const dim3 grid((unsigned)chunks);
      DG_CUDA(launch_kernel(scan_reduce, grid, kScanBlock, s, true, hist, hist_len, sums));
      DG_CUDA(launch_kernel(scan_spine, dim3(1), kScanBlock, s, true, sums, 1, chunks));
      DG_CUDA(launch_kernel(scan_apply, grid, kScanBlock, s, true, hist, hist_len, sums));
      count_launches(3);
    }
    if (csc && p == passes - 1) {
      // no keys are written: their place takes the table of rows
      uint4* table = reinterpret_cast<uint4*>(keys_out);
      DG_CUDA(cudaMemsetAsync(table, 0, (size_t)((count + 31) / 32) * sizeof(uint4), s));
      DG_CUDA(launch_kernel(row_table_kernel, dim3((unsigned)((g->row_plan.count + 7) / 8)), 256, s, true,
                            g->row_plan.chunks, g->row_plan.count, g->rowptr, csc->n, csc->columns, table));
      count_launches(1);
      csc->table = table;
    }
    DG_CUDA(launch_kernel(csc && p == passes - 1 ? digit_scatter<BITS, true> : digit_scatter<BITS, false>,
                          dim3((unsigned)tiles), kSortBlock, smem, s, true, keys_in, vals_in, count, shift, tiles, hist,
                          keys_out, vals_out, csc ? *csc : CscArgs{}));
    count_launches(2);
    keys_in = keys_out;
    vals_in = vals_out;
  }
  *sorted_keys = keys_in;
  return DG_OK;
}

// Stable LSD radix sort of `count` (key, value) pairs.  vals_in == nullptr means "the value of key
// i is i".  keys_in is only read; the sorted keys end in one of keys_buf (reported through
// *sorted_keys; keys_in may be keys_buf[1], which is first written by the second pass), the
// sorted values in vals_final (vals_tmp is the other buffer of the ping-pong).
static dg_status_t sort_run(const uint32_t* keys_in, const uint32_t* vals_in, int64_t count, SortPlan plan,
                            uint32_t* const keys_buf[2], uint32_t* vals_final, uint32_t* vals_tmp, uint32_t* hist,
                            uint32_t* sums, const uint32_t** sorted_keys, CscArgs* csc,
                            const Graph* g, cudaStream_t s) {
  if (plan.digit_bits == 9)
    return sort_passes_run<9>(keys_in, vals_in, count, plan.passes, keys_buf, vals_final, vals_tmp,
                              hist, sums, sorted_keys, csc, g, s);
  return sort_passes_run<8>(keys_in, vals_in, count, plan.passes, keys_buf, vals_final, vals_tmp,
                            hist, sums, sorted_keys, csc, g, s);
}
dg_status_t sort_pairs(const uint32_t* keys_in, const uint32_t* vals_in, int64_t count,
                       SortPlan plan, uint32_t* const keys_buf[2], uint32_t* vals_final,
                       uint32_t* vals_tmp, uint32_t* hist, uint32_t* sums,
                       const uint32_t** sorted_keys, cudaStream_t s) {
  return sort_run(keys_in, vals_in, count, plan, keys_buf, vals_final, vals_tmp, hist, sums, sorted_keys, nullptr,
                  nullptr, s);
}

// ptr[u] = first position whose sorted key is >= u, for u = 0..n (ptr[n] = count)
dg_status_t pointers_from_sorted_keys(const uint32_t* sorted, int64_t count, int64_t n,
                                      int64_t* ptr, cudaStream_t s) {
  DG_CUDA(cudaMemsetAsync(ptr, 0xFF, (size_t)(n + 1) * sizeof(int64_t), s));  // -1 everywhere
  const unsigned blocks = (unsigned)(((count + kColptrItems) / kColptrItems + 255) / 256);
  colptr_from_sorted_keys<<<blocks, 256, 0, s>>>(sorted, count, n, aligned16(sorted), ptr);
  DG_CUDA(cudaGetLastError());
  fill_long_gaps<<<(unsigned)((n + 1 + 255) / 256), 256, 0, s>>>(sorted, count, n, ptr);
  DG_CUDA(cudaGetLastError());
  count_launches(2);
  return DG_OK;
}

// out[k] = map[r] (r itself when map is nullptr) for the CSR row r that contains position k
dg_status_t expand_rows(const int64_t* rowptr, int64_t n, int64_t nnz, const int32_t* map,
                        uint32_t* out, cudaStream_t s) {
  if (nnz == 0) return DG_OK;
  const unsigned blocks = (unsigned)(((nnz + kRowItems - 1) / kRowItems + 255) / 256);
  expand_rows_kernel<<<blocks, 256, 0, s>>>(rowptr, n, nnz, map, out);
  DG_CUDA(cudaGetLastError());
  count_launches(1);
  return DG_OK;
}

void transpose_sizes(int64_t n, int64_t nnz, bool weighted, size_t* csc_bytes,
                     size_t* scratch_bytes) {
  const Layout L = make_layout(n, nnz, weighted);
  *csc_bytes = L.csc_bytes;
  *scratch_bytes = L.scratch_bytes;
}

static dg_status_t gather_weights(Graph* g, bool tabulated, cudaStream_t s) {
  if (g->nnz == 0 || !g->edge_w) return DG_OK;
  DG_CUDA(launch_kernel(tabulated ? gather_weights_kernel<true> : gather_weights_kernel<false>,
                        dim3((unsigned)((g->nnz + 1023) / 1024)), 256, s, true,
                        reinterpret_cast<const uint32_t*>(g->perm), g->nnz, g->edge_w, g->rowidx_T, g->rowptr,
                        g->self_loops_in_csc ? 1 : 0, const_cast<float*>(g->w_T),
                        const_cast<float*>(g->mean_scale_T)));
  count_launches(1);
  return DG_OK;
}
dg_status_t refresh_csc_weights(Graph* g, cudaStream_t s) { return gather_weights(g, false, s); }

dg_status_t transpose_run(Graph* g, void* csc, void* scratch, cudaStream_t s) {
  const int64_t n = g->n, nnz = g->nnz;
  const bool weighted = g->edge_w != nullptr;
  const Layout L = make_layout(n, nnz, weighted);
  char* cb = static_cast<char*>(csc);
  char* sb = static_cast<char*>(scratch);
  int64_t* colptr = reinterpret_cast<int64_t*>(cb + L.colptr_off);
  int32_t* rowidx_T = reinterpret_cast<int32_t*>(cb + L.rowidx_off);
  uint32_t* perm = reinterpret_cast<uint32_t*>(cb + L.perm_off);
  float* w_T = weighted ? reinterpret_cast<float*>(cb + L.w_off) : nullptr;
  float* mean_scale_T = reinterpret_cast<float*>(cb + L.mscale_off);
  uint32_t* keys_buf[2] = {reinterpret_cast<uint32_t*>(sb + L.keys_a_off),
                           reinterpret_cast<uint32_t*>(sb + L.keys_b_off)};
  uint32_t* vals_tmp = reinterpret_cast<uint32_t*>(sb + L.vals_off);
  uint32_t* hist = reinterpret_cast<uint32_t*>(sb + L.hist_off);
  uint32_t* sums = reinterpret_cast<uint32_t*>(sb + L.sums_off);

  if (nnz == 0) {
    DG_CUDA(cudaMemsetAsync(colptr, 0, (size_t)(n + 1) * 8, s));
  } else {
    const SortPlan plan = sort_plan(n);
    CscArgs c{nullptr, g->rowptr, n, reinterpret_cast<uint2*>(colptr), rowidx_T, mean_scale_T};
    columns_begin_kernel<<<(unsigned)(n / 256 + 1), 256, 0, s>>>(g->rowptr, n, g->self_loops ? 1 : 0, c.columns);
    DG_CUDA(cudaGetLastError());
    count_launches(1);
    const uint32_t* sorted = nullptr;
    if (dg_status_t st = sort_run(reinterpret_cast<const uint32_t*>(g->colidx), nullptr, nnz, plan, keys_buf, perm,
                                  vals_tmp, hist, sums, &sorted, &c, g, s))
      return st;
    const unsigned chunks = (unsigned)(n / kScanChunk + 1);  // of n + 1 columns
    if (n + 1 <= kFewEntries) {
      DG_CUDA(launch_kernel(scan_few<true>, dim3(1), kFewThreads, s, true, reinterpret_cast<uint32_t*>(c.columns), n + 1));
      count_launches(1);
    } else {
      DG_CUDA(launch_kernel(columns_reduce, dim3(chunks), kScanBlock, s, true, c.columns, n + 1));
      DG_CUDA(launch_kernel(scan_spine, dim3(1), kScanBlock, s, true, &c.columns->y, 2 * kScanChunk, chunks));
      DG_CUDA(launch_kernel(columns_apply, dim3(chunks), kScanBlock, s, true, c.columns, n + 1));
      count_launches(3);
    }
  }
  g->colptr = colptr;
  g->rowidx_T = rowidx_T;
  g->perm = reinterpret_cast<const int32_t*>(perm);
  g->w_T = w_T;
  g->mean_scale_T = mean_scale_T;
  g->self_loops_in_csc = g->self_loops;
  if (dg_status_t st = gather_weights(g, true, s)) return st;
  g->split_csc = nullptr;
  if (wants_split(n, nnz)) {
    // the columns come out of the stable sort ordered by row, so the check never fires here
    int32_t* split = reinterpret_cast<int32_t*>(cb + L.split_off);
    if (dg_status_t st = build_split(colptr, rowidx_T, n, g->fine_rows, split, g->counters + kUnsorted,
                                       nullptr, s))
      return st;
    g->split_csc = split;
  }
  return DG_OK;
}

}  // namespace dg
