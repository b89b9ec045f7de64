// scan.cu -- exclusive scans.
//
// The cell offsets of the bucket matrix (single pass), the per-minibatch
// offsets of the new nodes of each (tile, minibatch) cell (column scans), and
// the scan of the tile compaction at load time and of the staged rows (two
// launches, no waiting between blocks).
#include <mutex>
#include <unordered_map>

#include "common.cuh"
#include "internal.h"

namespace agnes {

namespace {

constexpr int kThreads = 256;
constexpr int kItems = 8;
constexpr int kChunk = kThreads * kItems;  // elements per block and chunk
constexpr int64_t kGridBlocks = 2048;      // blocks of a two-launch scan at most

// Exclusive block-wide scan of one int64 per thread; *total gets the sum.
__device__ __forceinline__ int64_t block_excl_scan(int64_t v, int64_t* total) {
  __shared__ int64_t warp_tot[kThreads / 32];
  __shared__ int64_t block_tot;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t incl = warp_incl_scan(v);
  if (lane == 31) warp_tot[warp] = incl;
  __syncthreads();
  if (warp == 0) {
    const int64_t w = lane < kThreads / 32 ? warp_tot[lane] : 0;
    const int64_t wi = warp_incl_scan(w);
    if (lane < kThreads / 32) warp_tot[lane] = wi - w;
    if (lane == kThreads / 32 - 1) block_tot = wi;
  }
  __syncthreads();
  const int64_t out = warp_tot[warp] + incl - v;
  *total = block_tot;
  __syncthreads();  // warp_tot / block_tot are reused by the next call
  return out;
}

// In-place exclusive scan of n int64 values, written by other blocks of the
// launch, by one CTA: each pass loads kItems consecutive values per thread before
// scanning them, so a pass costs one memory round trip.  Returns the total.
__device__ __forceinline__ int64_t cta_scan_inplace(int64_t* p, int64_t n) {
  int64_t carry = 0;
  for (int64_t base = 0; base < n; base += (int64_t)kThreads * kItems) {
    const int64_t i0 = base + (int64_t)threadIdx.x * kItems;
    int64_t v[kItems];
#pragma unroll
    for (int k = 0; k < kItems; ++k) v[k] = i0 + k < n ? *(volatile int64_t*)(p + i0 + k) : 0;
    int64_t run = 0;
#pragma unroll
    for (int k = 0; k < kItems; ++k) {
      const int64_t x = v[k];
      v[k] = run;
      run += x;
    }
    int64_t tot;
    const int64_t ex = block_excl_scan(run, &tot);
#pragma unroll
    for (int k = 0; k < kItems; ++k)
      if (i0 + k < n) p[i0 + k] = carry + ex + v[k];
    carry += tot;
  }
  return carry;
}

// Chunk sums; the last chunk to finish (atomic ticket after a fence, no waiting)
// then scans them in place, writes the total to out[n], and resets the ticket for
// the next scan.  A block takes chunks blockIdx.x, blockIdx.x + gridDim.x, ...
template <typename InT>
__global__ void __launch_bounds__(kThreads)
scan_reduce_kernel(const InT* __restrict__ in, int64_t n, int64_t chunks,
                   int64_t* __restrict__ partial, unsigned int* __restrict__ ticket,
                   int32_t* __restrict__ out, const int32_t* status) {
  grid_dep_wait();
  if (status && failed(status)) return;
  __shared__ int64_t wsum[kThreads / 32];
  __shared__ bool last;
  for (int64_t c = blockIdx.x; c < chunks; c += gridDim.x) {
    const int64_t begin = c * kChunk;
    int64_t sum = 0;
    InT v[kItems];  // all of the thread's loads in flight at once
#pragma unroll
    for (int k = 0; k < kItems; ++k) {
      const int64_t i = begin + k * kThreads + threadIdx.x;
      v[k] = i < n ? in[i] : (InT)0;
    }
#pragma unroll
    for (int k = 0; k < kItems; ++k) sum += (int64_t)v[k];
    sum = warp_sum(sum);
    if ((threadIdx.x & 31) == 0) wsum[threadIdx.x >> 5] = sum;
    __syncthreads();
    if (threadIdx.x < 32) {
      int64_t w = threadIdx.x < kThreads / 32 ? wsum[threadIdx.x] : 0;
      w = warp_sum(w);
      if (threadIdx.x == 0) {
        partial[c] = w;
        __threadfence();
        last = atomicAdd(ticket, 1u) == (unsigned)(chunks - 1);
      }
    }
    __syncthreads();
    if (last) {  // the final chunk: no later chunk of this block remains
      __threadfence();
      const int64_t carry = cta_scan_inplace(partial, chunks);
      if (threadIdx.x == 0) {
        out[n] = (int32_t)carry;
        *ticket = 0;
      }
    }
    __syncthreads();  // wsum and last are rewritten by the next chunk
  }
}

// Each warp scans 256 consecutive elements as 8 coalesced 32-wide slices
// (carry passed slice to slice), then the warps' totals are scanned.
template <typename InT>
__global__ void __launch_bounds__(kThreads)
scan_down_kernel(const InT* __restrict__ in, int32_t* __restrict__ out, int64_t n,
                 const int64_t* __restrict__ partial, const int32_t* status) {
  grid_dep_wait();
  if (status && failed(status)) return;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  __shared__ int64_t wtot[kThreads / 32];
  for (int64_t c = blockIdx.x; c * kChunk < n; c += gridDim.x) {
    const int64_t wbase = c * kChunk + (int64_t)warp * (32 * kItems);
    const int64_t chunk_off = partial[c];  // issued with the loads below
    int64_t v[kItems];
#pragma unroll
    for (int k = 0; k < kItems; ++k) {
      const int64_t i = wbase + k * 32 + lane;
      v[k] = i < n ? (int64_t)in[i] : 0;
    }
    int64_t carry = 0;
#pragma unroll
    for (int k = 0; k < kItems; ++k) {
      const int64_t inc = warp_incl_scan(v[k]);
      const int64_t x = v[k];
      v[k] = carry + inc - x;
      carry += __shfl_sync(0xffffffffu, inc, 31);
    }
    if (lane == 0) wtot[warp] = carry;
    __syncthreads();
    if (warp == 0) {
      const int64_t w = lane < kThreads / 32 ? wtot[lane] : 0;
      const int64_t wi = warp_incl_scan(w);
      if (lane < kThreads / 32) wtot[lane] = wi - w;
    }
    __syncthreads();
    const int64_t off = chunk_off + wtot[warp];
#pragma unroll
    for (int k = 0; k < kItems; ++k) {
      const int64_t i = wbase + k * 32 + lane;
      if (i < n) out[i] = (int32_t)(off + v[k]);
    }
    __syncthreads();  // wtot is rewritten by the next chunk
  }
}

// ---- single-pass flat scan (decoupled look-back) ----------------------------------
//
// Merrill & Garland's single-pass prefix scan (2016): every CTA takes the next
// tile of kFlatTile elements from a counter, publishes its tile's sum, and
// derives its exclusive prefix by walking back over its predecessors' flags
// until it meets an inclusive prefix; it then publishes that as well.  CTAs
// take tiles in the order they start, so a CTA waits only on tiles of CTAs
// that are already running; each wait is still bounded (kFlatSpinLimit
// polls), after which the CTA records kErrWaitTimeout and carries on.
//
// Scratch (uint64, zero between scans): [0] tile counter, [1] finished
// CTAs, [2 + t] flag of tile t = state << 62 | value, state 1 = the tile's
// sum, 2 = the inclusive prefix through the tile.  The last CTA to finish
// clears the flags and the counters.
constexpr int kFlatItems = 16;  // consecutive elements per thread (four 16-byte vectors)
constexpr int64_t kFlatTile = (int64_t)kThreads * kFlatItems;
constexpr unsigned long long kFlagAgg = 1ull << 62;
constexpr unsigned long long kFlagInc = 2ull << 62;
constexpr unsigned long long kFlagVal = (1ull << 62) - 1;
constexpr int kFlatSpinLimit = 1 << 20;

__device__ __forceinline__ unsigned long long flag_load(const unsigned long long* p) {
  return *(const volatile unsigned long long*)p;
}

__device__ __forceinline__ void flat_scan_cta(int32_t* __restrict__ in, int32_t* __restrict__ out,
                                              int64_t n, int64_t ntiles, bool clear,
                                              unsigned long long* scratch, int32_t* status) {
  // no early return on a failed status: every CTA takes its tile and counts
  // itself finished, so the scratch is left zero for the next scan
  __shared__ int64_t s_tile, s_excl;
  __shared__ int64_t warp_tot[kThreads / 32];
  __shared__ bool s_last;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  unsigned long long* flags = scratch + 2;
  if (tid == 0) {
    const int64_t t = (int64_t)atomicAdd(scratch, 1ull);
    if (t == ntiles - 1) scratch[0] = 0;  // every CTA has taken its tile
    s_tile = t;
  }
  __syncthreads();
  const int64_t tile = s_tile;
  // the thread's 16 consecutive elements
  const int64_t i0 = tile * kFlatTile + (int64_t)tid * kFlatItems;
  int32_t v[kFlatItems];
  if (i0 + kFlatItems <= n) {
    const int4* p = reinterpret_cast<const int4*>(in + i0);
#pragma unroll
    for (int q = 0; q < kFlatItems / 4; ++q) {
      const int4 x = p[q];
      v[4 * q] = x.x;
      v[4 * q + 1] = x.y;
      v[4 * q + 2] = x.z;
      v[4 * q + 3] = x.w;
    }
  } else {
#pragma unroll
    for (int k = 0; k < kFlatItems; ++k) v[k] = i0 + k < n ? in[i0 + k] : 0;
  }
  if (clear) {  // the counts start from zero next time, without a memset of their own
    if (i0 + kFlatItems <= n) {
      int4* p = reinterpret_cast<int4*>(in + i0);
#pragma unroll
      for (int q = 0; q < kFlatItems / 4; ++q) p[q] = make_int4(0, 0, 0, 0);
    } else {
#pragma unroll
      for (int k = 0; k < kFlatItems; ++k)
        if (i0 + k < n) in[i0 + k] = 0;
    }
  }
  int64_t mine = 0;
#pragma unroll
  for (int k = 0; k < kFlatItems; ++k) mine += v[k];
  // block scan of the threads' sums
  const int64_t incl = warp_incl_scan(mine);
  if (lane == 31) warp_tot[warp] = incl;
  __syncthreads();
  if (warp == 0) {
    const int64_t w = lane < kThreads / 32 ? warp_tot[lane] : 0;
    const int64_t wi = warp_incl_scan(w);
    if (lane < kThreads / 32) warp_tot[lane] = wi - w;
    const int64_t agg = __shfl_sync(0xffffffffu, wi, kThreads / 32 - 1);
    // publish, look back, publish the inclusive prefix
    int64_t excl = 0;
    if (tile == 0) {
      if (lane == 0) atomicExch(flags, kFlagInc | (unsigned long long)agg);
    } else {
      if (lane == 0) atomicExch(flags + tile, kFlagAgg | (unsigned long long)agg);
      for (int64_t j = tile - 1;; j -= 32) {
        const int64_t idx = j - lane;  // lane 0 the nearest predecessor
        unsigned long long f = kFlagInc;  // before tile 0: an inclusive prefix of 0
        if (idx >= 0) {
          f = flag_load(flags + idx);
          for (int spin = 0; (f >> 62) == 0; ++spin) {
            if (spin == kFlatSpinLimit) {
              atomicOr(status, kErrWaitTimeout);
              f = kFlagInc;
              break;
            }
            __nanosleep(64);
            f = flag_load(flags + idx);
          }
        }
        const unsigned inc = __ballot_sync(0xffffffffu, (f >> 62) == 2);
        const int stop = inc ? __ffs(inc) - 1 : 31;  // lanes 0 .. stop contribute
        excl += warp_sum(lane <= stop ? (int64_t)(f & kFlagVal) : (int64_t)0);
        if (inc) break;
      }
      if (lane == 0) atomicExch(flags + tile, kFlagInc | (unsigned long long)(excl + agg));
    }
    if (lane == 0) {
      s_excl = excl;
      if (tile == ntiles - 1) out[n] = (int32_t)(excl + agg);
    }
  }
  __syncthreads();
  int64_t run = s_excl + warp_tot[warp] + incl - mine;
  int32_t o[kFlatItems];
#pragma unroll
  for (int k = 0; k < kFlatItems; ++k) {
    o[k] = (int32_t)run;
    run += v[k];
  }
  if (i0 + kFlatItems <= n) {
    int4* p = reinterpret_cast<int4*>(out + i0);
#pragma unroll
    for (int q = 0; q < kFlatItems / 4; ++q)
      p[q] = make_int4(o[4 * q], o[4 * q + 1], o[4 * q + 2], o[4 * q + 3]);
  } else {
#pragma unroll
    for (int k = 0; k < kFlatItems; ++k)
      if (i0 + k < n) out[i0 + k] = o[k];
  }
  // the last CTA to finish (all look-backs done) clears the scratch
  if (tid == 0) {
    __threadfence();
    s_last = atomicAdd(scratch + 1, 1ull) == (unsigned long long)(ntiles - 1);
  }
  __syncthreads();
  if (s_last) {
    for (int64_t t = tid; t < ntiles; t += kThreads) flags[t] = 0;
    if (tid == 0) scratch[1] = 0;
  }
}

__global__ void __launch_bounds__(kThreads)
flat_scan_kernel(int32_t* __restrict__ in, int32_t* __restrict__ out, int64_t n, bool clear,
                 unsigned long long* scratch, int32_t* status) {
  grid_dep_wait();
  flat_scan_cta(in, out, n, gridDim.x, clear, scratch, status);
}

// ---- the scans between a hop's cells and its compaction -----------------------------
//
// The flat scan of the next frontier's cell counts, and exclusive scans down
// the columns of row-major [rows x cols] count matrices (one or two), in two
// launches: the first holds the flat scan's CTAs and the CTAs that sum the
// matrices' chunks of rows; in the second, each CTA adds up the sums of the
// chunks before its own and writes its chunk's prefixes.  Both are latency-
// bound (a few MB at most), so what counts is launches and dependent loads:
// the column scan used to be three launches on a side stream beside the flat
// scan, with an event to fork and one to join (16 x 1024 targets at [15, 10, 5]
// on 10M nodes: 638 -> 623 us a hyperbatch, the col fix-up moved into the
// compaction's launch; 128 x 1024 with three layers 5.27 -> 5.26 ms).
//
// A CTA covers `width` columns (the power of two from cols up, at most
// kColWidth) and kThreads / width groups of `depth` rows; depth grows with
// rows so that a column has at most kColChunks chunks, whose sums the second
// launch reads again in every CTA.
constexpr int kColWidth = 128;
constexpr int kColBatch = 16;  // rows whose loads are in flight together
constexpr int kColChunks = 256;

struct ColShape {
  int64_t rows;
  int32_t cols, width, depth, chunks, col_blocks;
};

ColShape col_shape(int64_t rows, int32_t cols) {
  ColShape s;
  s.rows = rows;
  s.cols = cols;
  s.width = 1;
  while (s.width < cols && s.width < kColWidth) s.width *= 2;
  const int64_t groups = kThreads / s.width;
  int64_t depth = (rows + groups * kColChunks - 1) / (groups * kColChunks);
  depth = (depth + kColBatch - 1) / kColBatch * kColBatch;
  s.depth = (int32_t)depth;
  s.chunks = (int32_t)((rows + groups * depth - 1) / (groups * depth));
  s.col_blocks = (cols + s.width - 1) / s.width;
  return s;
}

// Sum of rows [r0, r1) of column c.
__device__ __forceinline__ int32_t col_sum(const int32_t* __restrict__ in, int32_t cols, int32_t c,
                                           int64_t r0, int64_t r1) {
  int32_t sum = 0;
  for (int64_t r = r0; r < r1; r += kColBatch) {
    int32_t v[kColBatch];
#pragma unroll
    for (int k = 0; k < kColBatch; ++k) v[k] = r + k < r1 ? in[(r + k) * cols + c] : 0;
#pragma unroll
    for (int k = 0; k < kColBatch; ++k) sum += v[k];
  }
  return sum;
}

// One CTA's block b of a matrix: its chunk, and the thread's group and column
// (c >= cols: none).
struct ColPlace {
  int32_t chunk, group, groups, c;
  int64_t r0, r1;
};

__device__ __forceinline__ ColPlace col_place(const ColShape& s, int32_t b) {
  ColPlace p;
  p.groups = kThreads / s.width;
  p.group = (int32_t)threadIdx.x / s.width;
  p.chunk = b / s.col_blocks;
  p.c = (b - p.chunk * s.col_blocks) * s.width + (int32_t)threadIdx.x % s.width;
  p.r0 = min(s.rows, ((int64_t)p.chunk * p.groups + p.group) * s.depth);
  p.r1 = min(s.rows, p.r0 + s.depth);
  return p;
}

// Exclusive prefix of v over the groups of the thread's column, and the
// column's total; s_v is kThreads words.
__device__ __forceinline__ int32_t group_excl(int32_t* s_v, int32_t v, int32_t width,
                                              int32_t group, int32_t groups, int32_t* total) {
  const int tid = threadIdx.x;
  __syncthreads();
  s_v[tid] = v;
  __syncthreads();
  for (int d = 1; d < groups; d <<= 1) {  // inclusive scan over the groups
    const int32_t x = group >= d ? s_v[tid - d * width] : 0;
    __syncthreads();
    s_v[tid] += x;
    __syncthreads();
  }
  *total = s_v[(groups - 1) * width + tid % width];
  return s_v[tid] - v;
}

struct ColScan {
  const int32_t* in;
  int32_t* out;
  const int32_t* add_in;  // cols, or null
  int32_t* total[2];      // cols, or null
  int32_t* partial;       // chunks x cols
};

struct CellScansArgs {
  int32_t* flat_in;
  int32_t* flat_out;
  int64_t flat_n;
  int32_t flat_tiles;
  unsigned long long* flat_scratch;
  int32_t* status;
  ColShape shape;
  int32_t col_ctas;  // CTAs per matrix
  ColScan m[2];
};

__global__ void __launch_bounds__(kThreads) cell_scans_kernel(CellScansArgs a) {
  grid_dep_wait();
  if ((int32_t)blockIdx.x < a.flat_tiles) {
    flat_scan_cta(a.flat_in, a.flat_out, a.flat_n, a.flat_tiles, false, a.flat_scratch, a.status);
    return;
  }
  if (cta_failed(a.status)) return;
  __shared__ int32_t s_v[kThreads];
  int32_t b = (int32_t)blockIdx.x - a.flat_tiles;
  const int32_t which = b / a.col_ctas;
  b -= which * a.col_ctas;
  const ColScan& m = a.m[which];
  const ColPlace p = col_place(a.shape, b);
  const bool has = p.c < a.shape.cols;
  const int32_t sum = has ? col_sum(m.in, a.shape.cols, p.c, p.r0, p.r1) : 0;
  int32_t total;
  group_excl(s_v, sum, a.shape.width, p.group, p.groups, &total);
  if (has && p.group == 0) m.partial[(int64_t)p.chunk * a.shape.cols + p.c] = total;
}

__global__ void __launch_bounds__(kThreads) cell_scans_down_kernel(CellScansArgs a) {
  grid_dep_wait();
  if (failed(a.status)) return;
  __shared__ int32_t s_v[kThreads];
  int32_t b = (int32_t)blockIdx.x;
  const int32_t which = b / a.col_ctas;
  b -= which * a.col_ctas;
  const ColScan& m = a.m[which];
  const ColPlace p = col_place(a.shape, b);
  const int32_t cols = a.shape.cols;
  const bool has = p.c < cols;
  // no overlap of in and out: the loads of later rows are issued ahead of the
  // stores of earlier ones (19.2 -> 11.4 us at 31,068 x 128)
  const int32_t* __restrict__ in = m.in;
  int32_t* __restrict__ out = m.out;
  // the chunks before this one, a contiguous share per group
  const int32_t share = (p.chunk + p.groups - 1) / p.groups;
  const int32_t s0 = min(p.chunk, p.group * share);
  const int32_t before =
      has ? col_sum(m.partial, cols, p.c, s0, min(p.chunk, s0 + share)) : 0;
  const int32_t sum = has ? col_sum(in, cols, p.c, p.r0, p.r1) : 0;
  int32_t base, total;
  group_excl(s_v, before, a.shape.width, p.group, p.groups, &base);
  int32_t run = base + group_excl(s_v, sum, a.shape.width, p.group, p.groups, &total);
  if (!has) return;
  if (p.chunk == a.shape.chunks - 1 && p.group == 0) {
    const int32_t t = base + total + (m.add_in ? m.add_in[p.c] : 0);
    if (m.total[0]) m.total[0][p.c] = t;
    if (m.total[1]) m.total[1][p.c] = t;
  }
  for (int64_t r = p.r0; r < p.r1; r += kColBatch) {
    int32_t v[kColBatch];
#pragma unroll
    for (int k = 0; k < kColBatch; ++k) v[k] = r + k < p.r1 ? in[(r + k) * cols + p.c] : 0;
#pragma unroll
    for (int k = 0; k < kColBatch; ++k) {
      if (r + k < p.r1) out[(r + k) * cols + p.c] = run;
      run += v[k];
    }
  }
}

}  // namespace

int64_t cell_scans_scratch_elems(int64_t rows, int32_t cols) {
  return 2 * (int64_t)col_shape(rows, cols).chunks * cols;
}

cudaError_t cell_scans(int64_t rows, int32_t cols, int32_t* counts, int32_t* offsets,
                       uint64_t* flat_scratch, const ColumnScan* scans, int32_t nscans,
                       int32_t* scratch, int32_t* status, cudaStream_t st) {
  CellScansArgs a;
  a.flat_in = counts;
  a.flat_out = offsets;
  a.flat_n = rows * cols;
  a.flat_tiles = (int32_t)((a.flat_n + kFlatTile - 1) / kFlatTile);
  a.flat_scratch = reinterpret_cast<unsigned long long*>(flat_scratch);
  a.status = status;
  a.shape = col_shape(rows, cols);
  a.col_ctas = a.shape.chunks * a.shape.col_blocks;
  for (int32_t i = 0; i < 2; ++i) {
    const ColumnScan& c = scans[i < nscans ? i : 0];
    a.m[i] = ColScan{c.in, c.out, c.add_in, {c.total[0], c.total[1]},
                     scratch + (int64_t)i * a.shape.chunks * cols};
  }
  const unsigned cta = (unsigned)(a.col_ctas * nscans);
  cell_scans_kernel<<<(unsigned)a.flat_tiles + cta, kThreads, 0, st>>>(a);
  cell_scans_down_kernel<<<cta, kThreads, 0, st>>>(a);
  return cudaGetLastError();
}

int resident_grid(const void* kernel, int threads, int num_sms) {
  static std::mutex mu;
  static std::unordered_map<const void*, int> per_sm_cache;
  int per_sm = 0;
  {
    std::lock_guard<std::mutex> lock(mu);
    auto it = per_sm_cache.find(kernel);
    if (it != per_sm_cache.end()) per_sm = it->second;
  }
  if (per_sm == 0) {
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, threads, 0) !=
            cudaSuccess ||
        per_sm < 1) {
      cudaGetLastError();
      per_sm = 1;
    }
    std::lock_guard<std::mutex> lock(mu);
    per_sm_cache[kernel] = per_sm;
  }
  return per_sm * num_sms;
}

int64_t scan_scratch_elems(int64_t n) {
  return 1 + (n > 0 ? (n + kChunk - 1) / kChunk : 1);  // the ticket, then the chunk sums
}

int64_t flat_scan_scratch_elems(int64_t max_n) {
  return 2 + (max_n + kFlatTile - 1) / kFlatTile + 1;
}

cudaError_t flat_scan(int32_t* in, int32_t* out, int64_t n, bool clear, uint64_t* scratch,
                      int32_t* status, cudaStream_t st) {
  if ((uintptr_t)in % 16 != 0 || (uintptr_t)out % 16 != 0) return cudaErrorInvalidValue;
  const int64_t ntiles = n > 0 ? (n + kFlatTile - 1) / kFlatTile : 1;
  if (ntiles > 0x7fffffff) return cudaErrorInvalidValue;
  flat_scan_kernel<<<(unsigned)ntiles, kThreads, 0, st>>>(
      in, out, n, clear, reinterpret_cast<unsigned long long*>(scratch), status);
  return cudaGetLastError();
}

template <typename InT>
cudaError_t scan(const InT* in, int32_t* out, int64_t n, int64_t* scratch, const int32_t* status,
                 cudaStream_t st) {
  const int64_t chunks = scan_scratch_elems(n) - 1;
  const unsigned grid = (unsigned)(chunks < kGridBlocks ? chunks : kGridBlocks);
  int64_t* partial = scratch + 1;
  scan_reduce_kernel<InT><<<grid, kThreads, 0, st>>>(in, n, chunks, partial,
                                                     (unsigned int*)scratch, out, status);
  scan_down_kernel<InT><<<grid, kThreads, 0, st>>>(in, out, n, partial, status);
  return cudaGetLastError();
}

template cudaError_t scan<int32_t>(const int32_t*, int32_t*, int64_t, int64_t*, const int32_t*,
                                   cudaStream_t);
template cudaError_t scan<uint8_t>(const uint8_t*, int32_t*, int64_t, int64_t*, const int32_t*,
                                   cudaStream_t);

}  // namespace agnes
