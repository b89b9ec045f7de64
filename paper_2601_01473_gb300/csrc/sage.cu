// sage.cu -- a GraphSAGE-mean layer over one sampled hop of every minibatch
// of the last hyperbatch: the consumer of the prepared blocks.  It is an
// instance of eq. (1) (Sec. 3.1): the aggregation is the mean of the
// in-neighbours' rows and the update is a fully connected layer with ReLU,
//
//   out_i = ReLU(W_self x_i + W_neigh mean_{(i,u) in hop} x_u + b).
//
// One persistent, warp-specialised kernel, one CTA per SM.  The dst rows of
// minibatch j form ceil(|dst_h| / R) tiles of R rows, R = 128 (the MMA's M) or
// less where that gives every SM a tile or the rows are heavy.  Per tile of a CTA:
//   index warps     stage the tile's indptr and neighbour positions (one
//                   contiguous run of col) in a ring of shared-memory slots, so
//                   that the chain indptr -> col -> row costs the producers one
//                   trip per round of neighbours, not three, and ask for the
//                   tile's rows in L2 while they are at it (as far as L2 holds them),
//                   so that the trip ends there;
//   producer warps  form the update's input A = [x_i | mean_i]: an item (row,
//                   8-feature chunk) per thread, its neighbours' chunks summed
//                   in fp32 with several loads in flight, rounded to fp16 into
//                   a stage of the shared-memory ring laid out as a tcgen05
//                   K-major operand;
//   the MMA warp    issues the tile's tcgen05.mma chain (M = 128, N = d_out,
//                   K = 16 each) into one of two TMEM accumulators;
//   epilogue warps  read the accumulator back with tcgen05.ld, add the bias,
//                   apply ReLU and store.  They load W into shared memory first.
// All stages overlap.  Every mbarrier wait is bounded (a second, mbarrier.cuh); on
// timeout the kernel records an error, frees its tensor memory and returns.
//
// Bound by the neighbour rows' loads and the instructions that sum them (61% of
// the issue slots, the tensor pipe nearly idle), so most warps are producers, and
// how much L1 their loads in flight find matters as much (sage_shape).
// Measured against a gather kernel that wrote A to memory and a GEMM that read
// it back: 24 x 8192 rows of up to 15 neighbours, d_in = d_out = 128 in fp16,
// 241 -> 160 us a call; 128 x 1024 targets at [15, 10, 5] on 40M nodes with
// three layers 5.25 -> 4.35 ms.  On the way there: lanes over rows instead of
// over a row's chunks kept the L1 data pipe 81% busy (a quarter warp's loads
// touched 8 lines) and gained nothing; 16 producer warps instead of 24 cost 8%
// of that model, 8 neighbours in flight instead of 5 cost 11% (registers).  The
// rows asked for in L2 ahead: the model's outermost layer (3.4M rows, 16M
// edges) 1.15 -> 1.01 ms, 5.2 TB/s; four or five index slots, further ahead,
// lose that again.  With this and the steps noted below the 24 x 8192 layer takes
// 128 us and the model 4.03 ms.
#include <cuda_fp16.h>

#include "../../include/agnes.h"
#include "common.cuh"
#include "internal.h"
#include "mbarrier.cuh"

namespace agnes {

namespace {

constexpr int kM = 128;              // dst rows per tile at most (the MMA's M)
// warps: 0-3 epilogue, 4 MMA, then the index warps, then the producers
constexpr int kMmaWarp = 4;
constexpr int kIdxWarps = 2;
constexpr int kIdxWarp0 = kMmaWarp + 1;
constexpr int kProdWarp0 = kIdxWarp0 + kIdxWarps;
constexpr int kProdWarps = 24;
constexpr int kSageThreads = 32 * (kProdWarp0 + kProdWarps);
// Index slots: row, validity and col facts of a tile, its indptr relative to
// the tile's first edge, and up to idx_cap neighbour positions.
constexpr int kIdxSlots = 3;  // of most layers, with two or three stages (sage_shape)
constexpr int kIdxCapMax = 4096;
constexpr int kMaxSlots = 6;
constexpr int kMaxStages = 6;
struct IdxHead {
  int32_t i0, rows, j, staged;
  const int32_t* col;  // the tile's first edge's neighbour position, in global memory
  int64_t pad;
  int32_t ptr[kM + 4];
};
static_assert(sizeof(IdxHead) % 16 == 0, "the slots stay 16-byte aligned");
// Shared memory that leaves L1 about 60 KB, which the producers' loads in flight
// take (24 warps, 5 x 512 bytes each): the next larger split of the SM's 256 KB
// leaves 28.
constexpr size_t kSageL1Smem = 195 * 1024;
// Neighbours' rows on their way to L2 (129 MB) ahead of the producers at most, by
// the mean: 0.7 of it.  Further ahead they push one another out before they are
// used.  786k dst rows, d_in = d_out = 128 in fp16, with / without: 73 MB ahead 344 /
// 361 us, 146 MB 699 / 556; d_in = 64: 75 MB 310 / 300, 112 MB 443 / 388; 160 -> 192:
// 47 MB 419 / 489, 93 MB 784 / 771.
constexpr double kSageAheadBytes = 91e6;
// Every CTA asks for at least this much shared memory, so no two CTAs
// share an SM (and its 512 tensor-memory columns).
constexpr size_t kSageMinSmem = 120 * 1024;

constexpr int32_t kSageTimeout = 1;  // error word

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}

// Byte offset of element (r, k) in a K-major no-swizzle operand of `rows`
// rows: core matrix (r / 8, k / 8) at ((k / 8) * rows / 8 + r / 8) * 128.
__host__ __device__ __forceinline__ uint32_t kmajor_off(int r, int k, int rows) {
  return (uint32_t)((((k >> 3) * (rows >> 3)) + (r >> 3)) * 128 + (r & 7) * 16 + (k & 7) * 2);
}

// Byte offset of the 16-byte chunk c (elements 8 c .. 8 c + 7) of row r in a
// K-major operand of `rows` rows with 128-byte swizzle: blocks of 64 elements
// (`rows` rows of 128 bytes each), a row's eight chunks permuted by the row.
__device__ __forceinline__ uint32_t swizzled_off(int r, int c, int rows) {
  return (uint32_t)((c >> 3) * (rows * 128) + r * 128 + (((c & 7) ^ (r & 7)) << 4));
}

// tcgen05 shared-memory matrix descriptor, no swizzle: start address, the
// byte distance between core matrices adjacent in K (leading) and in M/N
// (stride), and the fixed version bits 46-48 = 0b001.
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr, uint32_t lbo, uint32_t sbo) {
  return (uint64_t)((addr & 0x3FFFF) >> 4) | ((uint64_t)((lbo & 0x3FFFF) >> 4) << 16) |
         ((uint64_t)((sbo & 0x3FFFF) >> 4) << 32) | (1ull << 46);
}

// The same for an operand with 128-byte swizzle (bits 61-63 = 2), its atoms of
// 8 rows x 128 bytes 1024 bytes apart; a K step within an atom starts 32 bytes
// on (the leading distance is not used).
__device__ __forceinline__ uint64_t smem_desc_swizzled(uint32_t addr) {
  return (uint64_t)((addr & 0x3FFFF) >> 4) | (1ull << 16) | ((uint64_t)(1024 >> 4) << 32) |
         (1ull << 46) | (2ull << 61);
}

// Instruction descriptor of kind::f16: fp32 accumulator (bits 4-5 = 1), fp16
// A and B (bits 7-9, 10-12 = 0), both K-major (bits 15, 16 = 0), N >> 3 at
// bits 17-22, M >> 4 at bits 24-28.
__device__ __forceinline__ uint32_t idesc_f16(int m, int n) {
  return (1u << 4) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(m >> 4) << 24);
}

__device__ __forceinline__ void mma_f16(uint32_t tmem_d, uint64_t a, uint64_t b, uint32_t idesc,
                                        uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
      :
      : "r"(tmem_d), "l"(a), "l"(b), "r"(idesc), "r"(accumulate)
      : "memory");
}

__device__ __forceinline__ void mma_commit(uint32_t bar) {
  asm volatile(
      "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar)
      : "memory");
}

// 8 consecutive features of a row as raw 16-byte vectors (one for fp16, two
// for fp32).
template <typename T>
struct Chunk {
  uint4 v[sizeof(T) / 2];
};

template <typename T>
__device__ __forceinline__ Chunk<T> load_chunk(const T* row, int c) {
  Chunk<T> ch;
#pragma unroll
  for (int q = 0; q < (int)(sizeof(T) / 2); ++q)
    ch.v[q] = __ldg((const uint4*)row + (sizeof(T) / 2) * c + q);
  return ch;
}

// Sums of the 8 features of a chunk as four pairs, added with the packed fp32
// add (each half rounded as by a single one).
struct Sum8 {
  uint64_t p[4];
};

__device__ __forceinline__ uint64_t pair(float a, float b) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}

__device__ __forceinline__ float2 unpair(uint64_t p) {
  float2 f;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(f.x), "=f"(f.y) : "l"(p));
  return f;
}

__device__ __forceinline__ void add_pair(uint64_t& acc, float a, float b) {
  asm("add.rn.f32x2 %0, %0, %1;" : "+l"(acc) : "l"(pair(a, b)));
}

__device__ __forceinline__ void add_chunk(const Chunk<__half>& ch, Sum8& acc) {
  const __half2* h = (const __half2*)&ch.v[0];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const float2 f = __half22float2(h[q]);
    add_pair(acc.p[q], f.x, f.y);
  }
}

__device__ __forceinline__ void add_chunk(const Chunk<float>& ch, Sum8& acc) {
  const float* f = (const float*)&ch.v[0];
#pragma unroll
  for (int q = 0; q < 4; ++q) add_pair(acc.p[q], f[2 * q], f[2 * q + 1]);
}

// a / b rounded to nearest, for r = 1 / b rounded to nearest: the estimate
// q = a r, corrected once by its exact remainder a - q b (Markstein, IBM J. Res.
// Dev. 34, 1990).  The remainder is exact unless it underflows, where |a / b| is
// below 2^-100 and fp16, what the quotient is rounded to next, keeps nothing of
// it; where q is not finite the remainder is no number, and q is the quotient.
__device__ __forceinline__ float quotient(float a, float b, float r) {
  const float q = a * r;
  const float rem = fmaf(-q, b, a);
  return rem == rem ? fmaf(rem, r, q) : q;
}

__device__ __forceinline__ uint4 to_half8(const float* f) {
  uint4 o;
  __half2 h;
  h = __floats2half2_rn(f[0], f[1]); o.x = *(uint32_t*)&h;
  h = __floats2half2_rn(f[2], f[3]); o.y = *(uint32_t*)&h;
  h = __floats2half2_rn(f[4], f[5]); o.z = *(uint32_t*)&h;
  h = __floats2half2_rn(f[6], f[7]); o.w = *(uint32_t*)&h;
  return o;
}

// 32 bytes of an output row: one store, a whole sector, where the output is
// 32-byte aligned.
__device__ __forceinline__ void store_sector(void* p, bool wide, uint4 a, uint4 b) {
  if (wide) {
    asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "r"(a.x),
                 "r"(a.y), "r"(a.z), "r"(a.w), "r"(b.x), "r"(b.y), "r"(b.z), "r"(b.w)
                 : "memory");
  } else {
    ((uint4*)p)[0] = a;
    ((uint4*)p)[1] = b;
  }
}

struct SageArgs {
  const void* x;              // minibatch j's src rows at x + (j * x_stride + r) * d_in
  int64_t x_stride;
  const int64_t* indptr;      // minibatch j at indptr + j * indptr_stride
  int64_t indptr_stride;
  const int32_t* col;
  int64_t col_stride;
  // the tiles of more than kInlineH minibatches, in device memory (else null:
  // SageTiles)
  const int32_t* tile_start;  // H + 1: first tile of each minibatch
  const int32_t* num_dst;     // H: |dst_h| per minibatch
  const int32_t* tile_mb;     // per tile: its minibatch
  int32_t H;
  int32_t total_tiles;
  int32_t d_in, d_out;
  int32_t tile_rows;          // R: dst rows per tile, a multiple of 8 up to kM
  uint64_t inv_chunks;        // ceil(2^32 / (d_in / 8))
  const __half* w;            // d_out x 2 d_in
  const float* bias;          // d_out or null
  void* out;                  // minibatch j's dst rows at out + (j * out_stride + i) * d_out
  int64_t out_stride;
  int32_t stages;             // A stages in shared memory
  int32_t slots;              // index slots
  bool ahead;                 // neighbours' rows are asked for in L2 ahead
  int32_t idx_cap;            // neighbour positions an index slot holds
  int32_t* err;
};

// The tiles of up to kInlineH minibatches travel with the launch: a tile's
// minibatch is found by a search in the parameters, instead of in tables that a
// copy would have to put on the device first (one layer of 300 to 18,000 rows:
// 64-81 -> 60-71 us a call).
constexpr int kInlineH = 256;
struct SageTiles {
  int32_t start[kInlineH + 1];  // first tile of each minibatch
  int32_t dst[kInlineH];        // |dst_h| of each minibatch
};

// Tile `tile`: its minibatch, first dst row, and the rows from there on.
struct SageTile {
  int32_t j, i0, rows;
};

__device__ __forceinline__ SageTile sage_tile(const SageArgs& a, const SageTiles& t,
                                              int32_t tile) {
  SageTile r;
  if (a.tile_mb) {
    r.j = __ldg(a.tile_mb + tile);
    r.i0 = (tile - __ldg(a.tile_start + r.j)) * a.tile_rows;
    r.rows = __ldg(a.num_dst + r.j) - r.i0;
  } else {
    int32_t lo = 0, hi = a.H;  // the last minibatch that starts at or before the tile
    while (hi - lo > 1) {
      const int32_t mid = (lo + hi) >> 1;
      if (t.start[mid] <= tile) lo = mid; else hi = mid;
    }
    r.j = lo;
    r.i0 = (tile - t.start[lo]) * a.tile_rows;
    r.rows = t.dst[lo] - r.i0;
  }
  return r;
}

// Shared memory: W and the A stages, the index slots, the mbarriers.  The MMA reads kM
// rows of every stage.  Where a stage has fewer, the others are whatever lies behind
// it, the next stage or W (8 KB at most, and W has as much: d_in > 64), and fill
// accumulator rows that nobody reads.  Stages of kM rows lie behind W.
struct SageSmem {
  uint8_t* w;
  uint8_t* a;
  uint8_t* idx;
  uint32_t idx_bytes;  // per slot
  uint64_t* bars;
};

__host__ __device__ __forceinline__ uint32_t idx_slot_bytes(int32_t idx_cap) {
  return (uint32_t)sizeof(IdxHead) + 4u * (uint32_t)idx_cap;  // idx_cap: a multiple of 4
}

template <int kRows>
__device__ __forceinline__ SageSmem sage_smem(uint8_t* smem, const SageArgs& a) {
  const uint32_t KT = 2 * a.d_in;
  SageSmem m;
  if (kRows == kM) {
    m.w = smem;
    m.a = m.w + (size_t)a.d_out * KT * 2;
    m.idx = m.a + (size_t)a.stages * kRows * KT * 2;
  } else {
    m.a = smem;
    m.w = m.a + (size_t)a.stages * kRows * KT * 2;
    m.idx = m.w + (size_t)a.d_out * KT * 2;
  }
  m.idx_bytes = idx_slot_bytes(a.idx_cap);
  m.bars = (uint64_t*)(m.idx + (size_t)a.slots * m.idx_bytes);
  return m;
}

// The mbarriers, as shared-memory addresses: full[s] / empty[s] of the A
// stages, dfull[d] / dempty[d] of the accumulators, ifull[q] / iempty[q] of
// the index slots, and W's.
struct SageBars {
  uint32_t base;
  __device__ uint32_t full(int s) const { return base + 8u * (uint32_t)s; }
  __device__ uint32_t empty(int s) const { return base + 8u * (uint32_t)(kMaxStages + s); }
  __device__ uint32_t dfull(int d) const { return base + 8u * (uint32_t)(2 * kMaxStages + d); }
  __device__ uint32_t dempty(int d) const { return base + 8u * (uint32_t)(2 * kMaxStages + 2 + d); }
  __device__ uint32_t ifull(int q) const { return base + 8u * (uint32_t)(2 * kMaxStages + 4 + q); }
  __device__ uint32_t iempty(int q) const {
    return base + 8u * (uint32_t)(2 * kMaxStages + 4 + kMaxSlots + q);
  }
  __device__ uint32_t w() const {
    return base + 8u * (uint32_t)(2 * kMaxStages + 4 + 2 * kMaxSlots);
  }
};
constexpr int kBars = 2 * kMaxStages + 4 + 2 * kMaxSlots + 1;
constexpr int kBarBytesNeeded = 8 * kBars + 8;  // and the TMEM address slot

// A walk around a ring of n slots: the slot of the current use, and its round.
struct Ring {
  int slot = 0, round = 0;
  __device__ void next(int n) {
    if (++slot == n) {
      slot = 0;
      ++round;
    }
  }
  // the parity of the phase that this use completes
  __device__ uint32_t parity() const { return (uint32_t)(round & 1); }
  // Whether this use may start: the use a round earlier has been released.
  __device__ bool free(uint32_t bar) const {
    return round == 0 || mbar_wait(bar, parity() ^ 1u);
  }
};

__device__ __forceinline__ void prefetch_l2(const void* p) {
  asm volatile("prefetch.global.L2 [%0];" ::"l"(p));
}

// An index warp: tiles w, w + kIdxWarps, ... of the CTA.
template <typename T>
__device__ __forceinline__ bool sage_index_warp(const SageArgs& a, const SageTiles& tiles,
                                                const SageSmem& m,
                                                const SageBars& bar, int w, int lane,
                                                int total_tiles) {
  Ring ring;
  for (int k = 0; k < w; ++k) ring.next(a.slots);
  for (int k = w;; k += kIdxWarps) {
    const int tile = (int)blockIdx.x + k * (int)gridDim.x;
    if (tile >= total_tiles) return true;
    const int q = ring.slot;
    if (!__all_sync(0xffffffffu, ring.free(bar.iempty(q)))) return false;
    IdxHead* h = (IdxHead*)(m.idx + (size_t)q * m.idx_bytes);
    int32_t* cols = (int32_t*)(h + 1);
    const SageTile st = sage_tile(a, tiles, tile);
    const int j = st.j, i0 = st.i0;
    const int rows = min(st.rows, a.tile_rows);
    const int64_t* ip = a.indptr + (size_t)j * a.indptr_stride + i0;
    const int64_t e0 = __ldg(ip);
    const int32_t n = (int32_t)(__ldg(ip + rows) - e0);
    for (int r = lane; r <= a.tile_rows; r += 32)
      h->ptr[r] = r < rows ? (int32_t)(__ldg(ip + r) - e0) : n;
    const int32_t* col = a.col + (size_t)j * a.col_stride + e0;
    const bool staged = n <= a.idx_cap;
    // the rows the tile reads -- its own, one after another, and its neighbours'
    // -- on their way to L2, up to `slots` tiles ahead of the producers
    const uint32_t row_bytes = (uint32_t)a.d_in * (uint32_t)sizeof(T);
    const char* x = (const char*)a.x + (size_t)j * a.x_stride * row_bytes;
    for (uint32_t b = 128u * lane; b < (uint32_t)rows * row_bytes; b += 4096)
      prefetch_l2(x + (size_t)i0 * row_bytes + b);
    if (staged) {
      for (int32_t i = lane; i < n; i += 256) {
        int32_t v[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) v[u] = i + 32 * u < n ? __ldg(col + i + 32 * u) : 0;
#pragma unroll
        for (int u = 0; u < 8; ++u)
          if (i + 32 * u < n) {
            cols[i + 32 * u] = v[u];
            if (a.ahead) {
              const char* row = x + (size_t)v[u] * row_bytes;
              for (uint32_t b = 0; b < row_bytes; b += 128) prefetch_l2(row + b);
            }
          }
      }
    }
    if (lane == 0) {
      h->i0 = i0;
      h->rows = rows;
      h->j = j;
      h->staged = staged;
      h->col = col;
    }
    __syncwarp();
    if (lane == 0) mbar_arrive(bar.ifull(q));
    for (int i = 0; i < kIdxWarps; ++i) ring.next(a.slots);
  }
}

// A producer warp: groups of 32 items of every tile of the CTA.
template <typename T, bool kSwizzle, int kRows>
__device__ __forceinline__ bool sage_producer_warp(const SageArgs& a, const SageSmem& m,
                                                   const SageBars& bar, int w, int lane,
                                                   int total_tiles) {
  constexpr int kER = sizeof(T) == 2 ? 5 : 3;  // neighbours in flight per item
  const int chunks = a.d_in / 8;
  const int groups = a.tile_rows * chunks / 32;
  const uint32_t stage_bytes = (uint32_t)(kRows * 4 * a.d_in);
  int first = w;  // the warp's first group, rotated from tile to tile so that a
                  // remainder of groups falls to every warp in turn
  // fp32's loads in flight leave no registers for the tile's and the slot's place,
  // which are computed anew (64 -> 128 on a skewed graph, fanouts 30 and 50, with this
  // and W first: 403 -> 389, 561 -> 543 us); in fp16 keeping them is faster
  constexpr bool kAnew = sizeof(T) == 4;
  Ring stage, slot;
  for (int k = 0, kept = blockIdx.x;; ++k, kept += kAnew ? 0 : gridDim.x, stage.next(a.stages)) {
    const int tile = kAnew ? (int)blockIdx.x + k * (int)gridDim.x : kept;
    if (tile >= total_tiles) return true;
    const int q = kAnew ? k % a.slots : slot.slot;
    const uint32_t parity = kAnew ? (uint32_t)((k / a.slots) & 1) : slot.parity();
    const bool ready = mbar_wait(bar.ifull(q), parity) && stage.free(bar.empty(stage.slot));
    if (!__all_sync(0xffffffffu, ready)) return false;
    const IdxHead* h = (const IdxHead*)(m.idx + (size_t)q * m.idx_bytes);
    const int32_t* cl = h->staged ? (const int32_t*)(h + 1) : h->col;
    const T* x = (const T*)a.x + (size_t)h->j * a.x_stride * a.d_in;
    const int32_t i0 = h->i0, rows = h->rows;
    uint8_t* A = m.a + stage.slot * stage_bytes;
    for (int g = first; g < groups; g += kProdWarps) {
      // the chunks fastest: the 8 lanes of a quarter warp, which one wavefront
      // serves, read one 128-byte line of a row
      const uint32_t item = (uint32_t)(g * 32 + lane);
      const int r = (int)((item * a.inv_chunks) >> 32);  // item / chunks
      const int c = (int)item - r * chunks;
      uint4 self = make_uint4(0, 0, 0, 0), mean = make_uint4(0, 0, 0, 0);
      if (r < rows) {
        const Chunk<T> sc = load_chunk<T>(x + (size_t)(i0 + r) * a.d_in, c);
        const int32_t e0 = h->ptr[r], e1 = h->ptr[r + 1];
        Sum8 acc;
#pragma unroll
        for (int z = 0; z < 4; ++z) acc.p[z] = 0;
        for (int32_t e = e0; e < e1; e += kER) {
          Chunk<T> val[kER];
#pragma unroll
          for (int u = 0; u < kER; ++u) {
            if (e + u < e1) {
              val[u] = load_chunk<T>(x + (size_t)cl[e + u] * a.d_in, c);
            } else {
#pragma unroll
              for (int z = 0; z < (int)(sizeof(T) / 2); ++z) val[u].v[z] = make_uint4(0, 0, 0, 0);
            }
          }
#pragma unroll
          for (int u = 0; u < kER; ++u) add_chunk(val[u], acc);
        }
        if constexpr (sizeof(T) == 2) {
          self = sc.v[0];
        } else {
          self = to_half8((const float*)&sc.v[0]);
        }
        if (e1 > e0) {
          const float deg = (float)(e1 - e0), inv = __frcp_rn(deg);
          float f[8];
#pragma unroll
          for (int z = 0; z < 4; ++z) {
            const float2 t = unpair(acc.p[z]);
            f[2 * z] = quotient(t.x, deg, inv);
            f[2 * z + 1] = quotient(t.y, deg, inv);
          }
          mean = to_half8(f);
        }
      }
      if constexpr (kSwizzle) {
        *(uint4*)(A + swizzled_off(r, c, kRows)) = self;
        *(uint4*)(A + swizzled_off(r, chunks + c, kRows)) = mean;
      } else {
        *(uint4*)(A + kmajor_off(r, c * 8, kRows)) = self;
        *(uint4*)(A + kmajor_off(r, a.d_in + c * 8, kRows)) = mean;
      }
    }
    first = (first + kProdWarps - groups % kProdWarps) % kProdWarps;
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    __syncwarp();
    if (lane == 0) {
      mbar_arrive(bar.full(stage.slot));
      mbar_arrive(bar.iempty(q));
    }
    if (!kAnew) slot.next(a.slots);
  }
}

// kSwizzle: A with 128-byte swizzle, where its rows are whole 64-element blocks
// (d_in a multiple of 32): a quarter warp's 8 chunks of one row then go to 8
// different bank groups.  Otherwise without swizzle, where they share one.
// kRows: the rows of a stage, tile_rows or more.
template <typename T, typename OutT, bool kSwizzle, int kRows>
__global__ void __launch_bounds__(kSageThreads, 1)
sage_kernel(SageArgs a, const __grid_constant__ SageTiles tiles) {
  extern __shared__ __align__(1024) uint8_t smem[];
  const int KT = 2 * a.d_in;
  const int N = a.d_out;
  const SageSmem m = sage_smem<kRows>(smem, a);
  const SageBars bar{smem_u32(m.bars)};
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const uint32_t ncols = 2 * N <= 64 ? 64 : (2 * N <= 128 ? 128 : (2 * N <= 256 ? 256 : 512));
  uint32_t* tmem_slot = (uint32_t*)(m.bars + kBars);

  // the swizzle's atoms are 1024-byte aligned: dynamic shared memory starts on
  // such a boundary, and W and a stage are multiples of that long
  if (kSwizzle && (smem_u32(smem) & 1023u) != 0) {
    if (tid == 0) *(volatile int32_t*)a.err = kSageTimeout;
    return;
  }
  if (warp == kMmaWarp) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(tmem_slot)),
                 "r"(ncols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  if (tid == 0) {
    for (int s = 0; s < kMaxStages; ++s) {
      mbar_init(bar.full(s), kProdWarps);
      mbar_init(bar.empty(s), 1);
    }
    for (int d = 0; d < 2; ++d) {
      mbar_init(bar.dfull(d), 1);
      mbar_init(bar.dempty(d), 4);  // one arrival per epilogue warp
    }
    for (int q = 0; q < kMaxSlots; ++q) {
      mbar_init(bar.ifull(q), 1);
      mbar_init(bar.iempty(q), kProdWarps);
    }
    mbar_init(bar.w(), 4);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *tmem_slot;
  const int total_tiles = a.total_tiles;
  bool ok = true;
  const bool wide_out = ((uintptr_t)a.out & 31) == 0;  // rows are whole 32-byte sectors

  if (warp >= kProdWarp0) {
    ok = sage_producer_warp<T, kSwizzle, kRows>(a, m, bar, warp - kProdWarp0, lane, total_tiles);
  } else if (warp >= kIdxWarp0) {
    ok = sage_index_warp<T>(a, tiles, m, bar, warp - kIdxWarp0, lane, total_tiles);
  } else if (warp == kMmaWarp) {
    // MMA issuer: each tile from the next stage into the next accumulator
    if (lane == 0) {
      const uint32_t idesc = idesc_f16(kM, N);
      const uint32_t w_addr = smem_u32(m.w);
      constexpr uint32_t kBlockBytes = kRows * 128;  // a swizzled 64-element block
      constexpr uint32_t kColBytes = kRows * 16;     // a core-matrix column
      const uint32_t stage_bytes = (uint32_t)(kRows * KT * 2);
      ok = mbar_wait(bar.w(), 0);
      Ring stage, acc;
      for (int tile = blockIdx.x; ok && tile < total_tiles; tile += gridDim.x) {
        const int s = stage.slot, d = acc.slot;
        if (!mbar_wait(bar.full(s), stage.parity()) || !acc.free(bar.dempty(d))) {
          ok = false;
          break;
        }
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const uint32_t a_addr = smem_u32(m.a) + (uint32_t)s * stage_bytes;
        const uint32_t dcol = tmem + (uint32_t)(d * N);
        // K step t covers K columns [16 t, 16 t + 16): core-matrix columns 2t, 2t+1
        for (int t = 0; t < KT / 16; ++t) {
          const uint64_t da =
              kSwizzle ? smem_desc_swizzled(a_addr + (uint32_t)(t >> 2) * kBlockBytes +
                                            (uint32_t)(t & 3) * 32)
                       : smem_desc(a_addr + (uint32_t)(2 * t) * kColBytes, kColBytes, 128);
          const uint64_t dw = smem_desc(w_addr + (uint32_t)(2 * t) * (uint32_t)(N / 8) * 128,
                                        (uint32_t)(N / 8) * 128, 128);
          mma_f16(dcol, da, dw, idesc, t > 0 ? 1u : 0u);
        }
        mma_commit(bar.empty(s));  // the stage is free once these MMAs have read it
        mma_commit(bar.dfull(d));  // and the accumulator is complete
        stage.next(a.stages);
        acc.next(2);
      }
    }
  } else {
    // W into its K-major layout: 16-byte chunk (n, kc) = W[n][8 kc .. 8 kc + 7]
    const int kchunks = KT / 8;
    for (int q = tid; q < N * kchunks; q += 128) {
      const int n = q / kchunks, kc = q - n * kchunks;
      *(uint4*)(m.w + kmajor_off(n, kc * 8, N)) = __ldg((const uint4*)(a.w + (size_t)n * KT) + kc);
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    __syncwarp();
    if (lane == 0) mbar_arrive(bar.w());
    // epilogue: warp w reads TMEM lanes 32 (w % 4) .. +31 (its rows)
    const int row = warp * 32 + lane;
    int k = 0;
    for (int tile = blockIdx.x; tile < total_tiles; tile += gridDim.x, ++k) {
      const int d = k & 1;
      if (!__all_sync(0xffffffffu, mbar_wait(bar.dfull(d), (uint32_t)((k / 2) & 1)))) {
        ok = false;
        break;
      }
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const SageTile st = sage_tile(a, tiles, tile);
      const bool valid = row < min(a.tile_rows, st.rows);
      OutT* orow = (OutT*)a.out + ((size_t)st.j * a.out_stride + st.i0 + row) * N;
      for (int c0 = 0; c0 < N; c0 += 32) {  // 32 columns per tcgen05.ld, one wait
        uint32_t v[32];
        const uint32_t taddr = tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)(d * N + c0);
        asm volatile(
            "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, "
            "%10, %11, %12, %13, %14, %15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, "
            "%26, %27, %28, %29, %30, %31}, [%32];"
            : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]),
              "=r"(v[6]), "=r"(v[7]), "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]),
              "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]), "=r"(v[16]), "=r"(v[17]),
              "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]),
              "=r"(v[24]), "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]),
              "=r"(v[30]), "=r"(v[31])
            : "r"(taddr)
            : "memory");
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
        if (valid) {
          uint4 half = make_uint4(0, 0, 0, 0);
#pragma unroll
          for (int g = 0; g < 4; ++g) {
            float f[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) {
              const int cc = c0 + 8 * g + q;
              f[q] = __uint_as_float(v[8 * g + q]) + (a.bias ? __ldg(a.bias + cc) : 0.f);
              f[q] = f[q] > 0.f ? f[q] : 0.f;
            }
            if constexpr (sizeof(OutT) == 4) {
              store_sector(orow + c0 + 8 * g, wide_out, *(const uint4*)&f[0],
                           *(const uint4*)&f[4]);
            } else if (g & 1) {
              store_sector(orow + c0 + 8 * (g - 1), wide_out, half, to_half8(f));
            } else {
              half = to_half8(f);
            }
          }
        }
      }
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      __syncwarp();
      if (lane == 0) mbar_arrive(bar.dempty(d));
    }
  }
  if (!ok) {
    *(volatile int32_t*)a.err = kSageTimeout;  // pinned host memory
    __threadfence_system();
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == kMmaWarp) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(ncols)
                 : "memory");
  }
}

// The rows of every tile from a.out, where the layer put them, to where they
// belong: a tile's rows are one contiguous run of row_vecs 16-byte vectors each in
// both.
__global__ void __launch_bounds__(256)
sage_place_kernel(SageArgs a, const __grid_constant__ SageTiles tiles, int32_t row_vecs,
                  uint4* __restrict__ out, int64_t out_stride) {
  const uint4* from = (const uint4*)a.out;
  for (int tile = blockIdx.x; tile < a.total_tiles; tile += gridDim.x) {
    const SageTile t = sage_tile(a, tiles, tile);
    const int32_t n = min(a.tile_rows, t.rows) * row_vecs;
    const uint4* src = from + ((size_t)t.j * a.out_stride + t.i0) * row_vecs;
    uint4* dst = out + ((size_t)t.j * out_stride + t.i0) * row_vecs;
    for (int32_t q = threadIdx.x; q < n; q += blockDim.x) dst[q] = src[q];
  }
}

// Shared memory of the kernel with `stages` A stages and index slots of
// idx_cap neighbour positions.
size_t sage_smem_bytes(int64_t d_in, int64_t d_out, int stages, int stage_rows, int slots,
                       int32_t idx_cap) {
  return (size_t)d_out * 2 * d_in * 2 + (size_t)stages * stage_rows * 2 * d_in * 2 +
         (size_t)slots * idx_slot_bytes(idx_cap) + kBarBytesNeeded;
}

// What the entry point's limit counts: W, kM rows of A and 128 bytes.  The largest
// accepted shapes (d_in a multiple of 8, d_out of 32) leave 2048 bytes of the
// limit or more, so the heads of the index slots (kIdxSlots * sizeof(IdxHead)
// = 1680 bytes) and the mbarriers with the TMEM address slot always fit beside them.
size_t stated_smem_bytes(int64_t d_in, int64_t d_out) {
  return (size_t)d_out * 2 * d_in * 2 + (size_t)kM * 2 * d_in * 2 + 128;
}
static_assert(kIdxSlots * sizeof(IdxHead) + kBarBytesNeeded <= 2048, "the largest shapes fit");

bool is_device_ptr(const void* p) {
  cudaPointerAttributes attr;
  if (cudaPointerGetAttributes(&attr, p) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return attr.type == cudaMemoryTypeDevice || attr.type == cudaMemoryTypeManaged;
}

// Whether [a, a + na) and [b, b + nb) share a byte (a null range has none).
bool ranges_overlap(const void* a, size_t na, const void* b, size_t nb) {
  return a && b && (uintptr_t)a < (uintptr_t)b + nb && (uintptr_t)b < (uintptr_t)a + na;
}

template <typename T, typename OutT, bool kSwizzle, int kRows>
cudaError_t launch_sage_typed(const SageArgs& a, const SageTiles& t, int num_sms,
                              cudaStream_t st) {
  size_t smem = sage_smem_bytes(a.d_in, a.d_out, a.stages, kRows, a.slots, a.idx_cap);
  if (smem < kSageMinSmem) smem = kSageMinSmem;
  const auto kernel = sage_kernel<T, OutT, kSwizzle, kRows>;
  cudaError_t e =
      cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  const int grid = a.total_tiles < num_sms ? a.total_tiles : num_sms;
  kernel<<<grid, kSageThreads, smem, st>>>(a, t);
  return cudaGetLastError();
}

template <typename T, typename OutT>
cudaError_t launch_sage(const SageArgs& a, const SageTiles& t, int stage_rows, int num_sms,
                        cudaStream_t st) {
  const bool swizzle = a.d_in % 32 == 0;
  const auto launch =
      stage_rows == kM ? (swizzle ? launch_sage_typed<T, OutT, true, kM>
                                  : launch_sage_typed<T, OutT, false, kM>)
                       : (swizzle ? launch_sage_typed<T, OutT, true, kM / 2>
                                  : launch_sage_typed<T, OutT, false, kM / 2>);
  return launch(a, t, num_sms, st);
}

// How a layer is cut into tiles and uses its shared memory.
struct SageShape {
  int tile_rows, stages, stage_rows, slots;
  int32_t idx_cap;
};

// What decides it.
struct SageLoad {
  int64_t d_in, d_out;
  int64_t row_bytes;  // of x
  double degree;      // mean edges per dst row
  int64_t fanout;     // the most
};

// Neighbour positions for which an index slot has room beside the rest, in `bytes`
// of shared memory (negative: the rest does not fit).
int32_t idx_room(const SageLoad& l, const SageShape& s, size_t bytes) {
  const size_t base = sage_smem_bytes(l.d_in, l.d_out, s.stages, s.stage_rows, s.slots, 0);
  if (base > bytes) return -1;
  return (int32_t)((bytes - base) / (sizeof(int32_t) * s.slots)) & ~3;
}

// The shape for tiles of up to tile_rows rows.
//
// What shared memory takes is not L1's, and the producers' loads in flight need L1,
// so more stages, rows in a stage and staged indices pay only up to a point, and
// that point depends on what a dst row costs the producers: the bytes of its own
// row and its neighbours', (1 + degree) * row_bytes.
//  - Light rows: tiles of 128, as the epilogue and the MMA cost the same for fewer.
//  - Heavy rows: tiles of 64 in two stages of 64 rows, which take what one stage of
//    128 does, so that they always fit.
//  - One stage of 128 rows, where two do not fit, only for light rows: the
//    producers wait for every tile's MMA.
//  - Up to 64 features two stages of 128 rows are small: always those.
// 786k dst rows of equal degree, us, tiles of 128 / 64 rows.  d_in = d_out = 128 in
// fp16: degree 3 262 / 298, 5 343 / 345, 8 485 / 414, 20 926 / 780; 3.5M rows of
// degree 4.75 on 40M nodes 1122 / 1260.  In fp32: degree 2 321 / 314, 3 436 / 354.
// 128 -> 192, whose two stages leave no room to stage indices: 3 311 / 333, 5 416 /
// 361.  128 -> 256, one stage: 1 335 / 371, 2 374 / 370, 3 424 / 392, 8 641 / 457.
// 64 -> 64: 3 199 / 237, 20 475 / 498.
// The same layers with up to three stages of 128 rows whatever the degree, before,
// and with two kernels, an aggregation at full occupancy and a GEMM, before that:
// 128 -> 128 at degree 12 882 and 835 (now 557), at 20 1337 and 1149 (781); 256 -> 64
// at 12 1776 and 1450 (1051); fp32 128 -> 128 at 12 1598 and 1160 (903).
SageShape sage_shape(const SageLoad& l, int32_t tile_rows) {
  SageShape s{tile_rows, 2, kM, kIdxSlots, 0};
  if (l.d_in > 64) {
    const int32_t room = idx_room(l, s, AGNES_SAGE_MAX_SMEM);
    const bool f32 = l.row_bytes > 2 * l.d_in;  // its loads take a fifth more of L1
    const double heavy = room < 0                 ? 2.4 * l.d_out
                         : room < kM * l.degree ? 1000
                         : f32                  ? 1300
                                                : 1800;
    if ((1 + l.degree) * l.row_bytes >= heavy) {
      s.stage_rows = kM / 2;
      s.tile_rows = tile_rows < kM / 2 ? tile_rows : kM / 2;
    } else if (room < 0) {
      s.stages = 1;
    }
  }
  // The slots stage twice a tile's mean of edges.  Rows of up to 48 bytes are read by
  // a thread or two an edge: staging costs the two index warps more than it saves
  // (8 -> 32 at degree 30: 474 us staged, 235 not; two kernels 292).
  int32_t want = 0;
  if (l.row_bytes > 48) {
    const double most = 2 * l.degree + 1 < l.fanout ? 2 * l.degree + 1 : l.fanout;
    want = (int32_t)(s.tile_rows * most < kIdxCapMax ? s.tile_rows * most + 3 : kIdxCapMax) & ~3;
  }
  // More stages and slots as long as L1 keeps its share: six where a tile is work
  // for a third of the producer warps, so that three tiles are in the making (8 -> 32
  // at degree 20: 224 -> 186 us), four up to 64 features (64 -> 64 on a skewed graph,
  // fanouts 15 and 50: 241 -> 232, 404 -> 383), else three.
  const int rings[][2] = {{6, 6}, {4, 4}, {3, kIdxSlots}};  // stages, slots
  const int groups = s.tile_rows * (int)l.d_in / 8 / 32;
  for (int i = 3 * groups <= kProdWarps ? 0 : l.d_in <= 64 ? 1 : 2; s.stages == 2 && i < 3; ++i) {
    SageShape more = s;
    more.stages = rings[i][0];
    more.slots = rings[i][1];
    if (idx_room(l, more, kSageL1Smem) >= want) s = more;
  }
  const int32_t room = idx_room(l, s, AGNES_SAGE_MAX_SMEM);
  s.idx_cap = room < want ? room : want;
  return s;
}

}  // namespace

}  // namespace agnes

using namespace agnes;

extern "C" agnes_status agnes_sage_mean_layer(agnes_ctx* ctx, int32_t hop, const void* x,
                                              int32_t x_dtype, int64_t x_stride_rows,
                                              int64_t d_in, const void* w, const float* bias,
                                              int32_t d_out, void* out, int32_t out_dtype,
                                              int64_t out_stride_rows, void* cuda_stream) {
  if (!ctx || !x || !w || !out) {
    ctx_set_error(ctx, "ctx, x, w and out must be non-NULL");
    return AGNES_EINVAL;
  }
  GraphView g;
  ctx_graph_view(ctx, &g);
  DeviceGuard dg(g.device);
  if (!dg.ok()) {
    ctx_set_error(ctx, "cudaSetDevice(%d) failed", g.device);
    return AGNES_ECUDA;
  }
  agnes_hyperbatch_view v;
  agnes_status rc = agnes_fetch_hyperbatch(ctx, &v);
  if (rc != AGNES_OK) return rc;
  if (hop < 0 || hop >= v.K) {
    ctx_set_error(ctx, "hop %d outside [0, %d)", hop, v.K);
    return AGNES_EINVAL;
  }
  if ((x_dtype != AGNES_F32 && x_dtype != AGNES_F16) ||
      (out_dtype != AGNES_F32 && out_dtype != AGNES_F16)) {
    ctx_set_error(ctx, "x_dtype and out_dtype must be AGNES_F32 or AGNES_F16");
    return AGNES_EINVAL;
  }
  if (d_in < 8 || d_in % 8 != 0 || d_out < 32 || d_out > 256 || d_out % 32 != 0) {
    ctx_set_error(ctx, "d_in must be a positive multiple of 8 and d_out a multiple of 32 in "
                       "[32, 256]");
    return AGNES_EINVAL;
  }
  if (stated_smem_bytes(d_in, d_out) > AGNES_SAGE_MAX_SMEM) {
    ctx_set_error(ctx, "d_in %lld with d_out %d needs %zu bytes of shared memory (limit %d)",
                  (long long)d_in, d_out, stated_smem_bytes(d_in, d_out), AGNES_SAGE_MAX_SMEM);
    return AGNES_ERANGE;
  }
  if (((uintptr_t)x | (uintptr_t)w | (uintptr_t)out) % 16 != 0 ||
      ((uintptr_t)bias % 4) != 0) {
    ctx_set_error(ctx, "x, w and out must be 16-byte aligned");
    return AGNES_EINVAL;
  }
  const int H = v.H;
  const int32_t* dst_size = v.node_size + (size_t)hop * H;
  // rows per tile: 128 (the MMA's M), halved down to 32 while that leaves SMs
  // without a tile -- a small layer is bound by the latency of its producers'
  // loads, and the MMA costs the same for fewer rows
  auto tiles_of = [&](int32_t rows) {
    int64_t n = 0;
    for (int j = 0; j < H; ++j) n += ((int64_t)dst_size[j] + rows - 1) / rows;
    return n;
  };
  int32_t tile_rows = kM;
  while (tile_rows > 32 && tiles_of(tile_rows) < g.num_sms) tile_rows /= 2;
  const int64_t fanout = v.col_stride[hop] / (v.indptr_stride[hop] - 1);
  const size_t x_row = (size_t)d_in * (x_dtype == AGNES_F32 ? 4 : 2);
  int64_t dsts_all = 0, srcs_all = 0, edges_all = 0;
  for (int j = 0; j < H; ++j) {
    dsts_all += dst_size[j];
    srcs_all += v.src_size[(size_t)hop * H + j];
    edges_all += v.edges[(size_t)hop * H + j];
  }
  const double degree = dsts_all > 0 ? (double)edges_all / dsts_all : 0;
  const SageShape shape =
      sage_shape(SageLoad{d_in, d_out, (int64_t)x_row, degree, fanout}, tile_rows);
  tile_rows = shape.tile_rows;
  int64_t tiles = tiles_of(tile_rows);
  int64_t max_src = 0, max_dst = 0;
  const bool inline_tiles = H <= kInlineH;
  // pinned staging: error word (16 bytes; the kernel writes it in place), then,
  // where the tiles do not travel with the launch, tile_start (H + 1), num_dst
  // (H), tile_mb (one per tile)
  const size_t tab_bytes =
      inline_tiles ? 0 : sizeof(int32_t) * ((size_t)2 * H + 1 + (size_t)tiles);
  void* hp = nullptr;
  cudaError_t e = ctx_pinned(ctx, 16 + tab_bytes, &hp);
  if (e != cudaSuccess) {
    ctx_set_error(ctx, "agnes_sage_mean_layer: %s", cudaGetErrorString(e));
    return AGNES_ENOMEM;
  }
  int32_t* h_err = (int32_t*)hp;
  int32_t* tabs = (int32_t*)((char*)hp + 16);
  SageTiles inl;
  int32_t* starts = inline_tiles ? inl.start : tabs;
  int32_t* dsts = inline_tiles ? inl.dst : tabs + H + 1;
  tiles = 0;
  for (int j = 0; j < H; ++j) {
    const int64_t nd = dst_size[j];
    const int64_t ns = v.src_size[(size_t)hop * H + j];
    max_dst = nd > max_dst ? nd : max_dst;
    max_src = ns > max_src ? ns : max_src;
    starts[j] = (int32_t)tiles;
    dsts[j] = (int32_t)nd;
    const int64_t nt = (nd + tile_rows - 1) / tile_rows;
    if (!inline_tiles)
      for (int64_t t = tiles; t < tiles + nt; ++t) tabs[2 * H + 1 + t] = j;
    tiles += nt;
  }
  starts[H] = (int32_t)tiles;
  if (x_stride_rows < max_src || out_stride_rows < max_dst) {
    ctx_set_error(ctx, "x_stride_rows must be >= %lld and out_stride_rows >= %lld",
                  (long long)max_src, (long long)max_dst);
    return AGNES_EINVAL;
  }
  if (!is_device_ptr(x) || !is_device_ptr(w) || !is_device_ptr(out) ||
      (bias && !is_device_ptr(bias))) {
    ctx_set_error(ctx, "x, w, bias and out must be device memory");
    return AGNES_EINVAL;
  }
  cudaStream_t st = (cudaStream_t)cuda_stream;
  // Tiles are stored while other CTAs still read the inputs, so an output that
  // shares memory with any of them (a layer in place) is formed in scratch and
  // placed once the kernel has read everything.
  const size_t out_row = (size_t)d_out * (out_dtype == AGNES_F32 ? 4 : 2);
  const size_t out_span = ((size_t)(H - 1) * out_stride_rows + max_dst) * out_row;
  auto out_meets = [&](const void* p, size_t bytes) {
    return ranges_overlap(out, out_span, p, bytes);
  };
  const bool staged =
      out_meets(x, ((size_t)(H - 1) * x_stride_rows + max_src) * x_row) ||
      out_meets(w, (size_t)d_out * 2 * d_in * sizeof(__half)) ||
      out_meets(bias, (size_t)d_out * sizeof(float)) ||
      out_meets(v.indptr[hop], (size_t)H * v.indptr_stride[hop] * sizeof(int64_t)) ||
      out_meets(v.col[hop], (size_t)H * v.col_stride[hop] * sizeof(int32_t));
  // the tables on the device, then the staged rows
  const size_t tab_room = (tab_bytes + 255) & ~(size_t)255;
  const size_t scratch_bytes = tab_room + (staged ? (size_t)H * max_dst * out_row : 0);
  void* scratch = nullptr;
  if (scratch_bytes > 0) e = ctx_scratch(ctx, scratch_bytes, &scratch);
  int32_t* d_tabs = (int32_t*)scratch;
  int32_t* d_err = nullptr;
  if (e == cudaSuccess) e = cudaHostGetDevicePointer((void**)&d_err, h_err, 0);
  *h_err = 0;
  if (e == cudaSuccess && !inline_tiles)
    e = cudaMemcpyAsync(d_tabs, tabs, tab_bytes, cudaMemcpyHostToDevice, st);
  if (e == cudaSuccess && tiles > 0) {
    SageArgs a;
    a.x = x;
    a.x_stride = x_stride_rows;
    a.indptr = v.indptr[hop];
    a.indptr_stride = v.indptr_stride[hop];
    a.col = v.col[hop];
    a.col_stride = v.col_stride[hop];
    a.tile_start = inline_tiles ? nullptr : d_tabs;
    a.num_dst = inline_tiles ? nullptr : d_tabs + H + 1;
    a.tile_mb = inline_tiles ? nullptr : d_tabs + 2 * H + 1;
    a.H = H;
    a.total_tiles = (int32_t)tiles;
    a.d_in = (int32_t)d_in;
    a.d_out = d_out;
    a.tile_rows = tile_rows;
    a.inv_chunks = ((1ull << 32) + d_in / 8 - 1) / (d_in / 8);
    a.w = (const __half*)w;
    a.bias = bias;
    a.out = staged ? (char*)scratch + tab_room : out;
    a.out_stride = staged ? max_dst : out_stride_rows;
    a.stages = shape.stages;
    a.slots = shape.slots;
    const int64_t ctas = tiles < g.num_sms ? tiles : g.num_sms;
    // the rows ahead: the edges' of the tiles in the slots, or, where fewer, all
    // rows of the minibatches that those tiles lie in
    const double rows_ahead = (double)ctas * shape.slots * tile_rows;
    const double near = (rows_ahead * H / dsts_all + 1) * srcs_all / H;
    a.ahead = (rows_ahead * degree < near ? rows_ahead * degree : near) * x_row <= kSageAheadBytes;
    a.idx_cap = shape.idx_cap;
    a.err = d_err;
    const auto launch =
        x_dtype == AGNES_F16
            ? (out_dtype == AGNES_F32 ? launch_sage<__half, float> : launch_sage<__half, __half>)
            : (out_dtype == AGNES_F32 ? launch_sage<float, float> : launch_sage<float, __half>);
    e = launch(a, inl, shape.stage_rows, g.num_sms, st);
    if (e == cudaSuccess && staged) {
      sage_place_kernel<<<fitted_grid((const void*)sage_place_kernel, 256, g.num_sms, tiles), 256,
                          0, st>>>(a, inl, (int32_t)(out_row / 16), (uint4*)out, out_stride_rows);
      e = cudaGetLastError();
    }
  }
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) {
    ctx_set_error(ctx, "agnes_sage_mean_layer: %s", cudaGetErrorString(e));
    return e == cudaErrorMemoryAllocation ? AGNES_ENOMEM : AGNES_ECUDA;
  }
  if (*(volatile int32_t*)h_err != 0) {
    ctx_set_error(ctx, "agnes_sage_mean_layer: a tensor-core or copy wait ran out");
    return AGNES_ETIMEOUT;
  }
  return AGNES_OK;
}
