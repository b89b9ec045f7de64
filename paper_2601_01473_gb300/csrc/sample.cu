// sample.cu -- bucketing of the targets and per-hop neighbour sampling.
//
// Bucket matrix (Sec. 3.4 (3), Algorithm 1's Bck_{i,j}): frontier entries are
// kept per (tile, minibatch) cell in tile-major, minibatch-minor order, sorted
// by node id inside a cell, each with its global output row
// g = j * capK + position.  A topology block's requests are therefore one
// contiguous run of the bucket, and sampling walks the bucket in order, so the
// block is read once for all minibatches of the hyperbatch (Sec. 3.3) and its
// adjacency data is reused out of L2.
//
// Sampling (Sec. 3.1, Algorithm 1's Sample): up to k neighbours per frontier
// node, uniformly without replacement; all of them in CSR order when
// deg <= k, else Floyd's algorithm (Bentley & Floyd, CACM 1987) with
// Philox4x32-10 draws keyed on (seed; v, hop, slot, g).  For k <= 32 a group
// of k lanes handles one frontier node (32 / k nodes per warp round): lane s
// draws slot s's candidate in parallel and the k-step collision resolution
// runs over warp shuffles.  Above 32 a warp takes 32 slots at a time,
// checking each candidate against the earlier chunks' choices (in shared
// memory up to kWideMax, in a hash set in global memory beyond).
#include "common.cuh"
#include "internal.h"

namespace agnes {

namespace {

constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;

// ---- bucketing of the targets ------------------------------------------------

// Counts the targets per (tile, minibatch) cell; rank[i] = the target's place
// among its cell's (the order of arrival).
__global__ void __launch_bounds__(kThreads)
targets_count_kernel(const int32_t* __restrict__ nodes, int64_t capK, int32_t H, int32_t B,
                     int32_t N, TileMap tm, int32_t* __restrict__ fcnt,
                     int32_t* __restrict__ rank, int32_t* status) {
  grid_dep_wait();
  const int64_t total = (int64_t)H * B;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t i0 = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) & ~31ll; i0 < total;
       i0 += stride) {
    const int64_t i = i0 + lane_id();
    bool active = i < total;
    int64_t cell = 0;
    if (active) {
      const int32_t j = (int32_t)(i / B);
      const int32_t v = nodes[j * capK + (i - (int64_t)j * B)];
      if (v < 0 || v >= N) {
        atomicOr(status, kErrTargetRange);
        active = false;
      } else {
        cell = (int64_t)tile_of(tm, v) * H + j;
      }
    }
    const unsigned mask = __ballot_sync(0xffffffffu, active);
    if (active) rank[i] = warp_agg_add(fcnt, cell, mask);
  }
}

// Every target to its cell's slots, in order of arrival.
__global__ void __launch_bounds__(kThreads)
targets_scatter_kernel(const int32_t* __restrict__ nodes, int64_t capK, int32_t H, int32_t B,
                       TileMap tm, const int32_t* __restrict__ fcell_off,
                       const int32_t* __restrict__ rank, int32_t* __restrict__ tmp_id,
                       int32_t* __restrict__ tmp_pos, const int32_t* status) {
  grid_dep_wait();
  if (failed(status)) return;
  const int64_t total = (int64_t)H * B;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < total; i += stride) {
    const int32_t j = (int32_t)(i / B);
    const int64_t pos = j * capK + (i - (int64_t)j * B);
    const int32_t v = nodes[pos];
    const int32_t slot = fcell_off[(int64_t)tile_of(tm, v) * H + j] + rank[i];
    tmp_id[slot] = v;
    tmp_pos[slot] = (int32_t)pos;
  }
}

// A cell of up to kWalkMax targets is ordered by a thread per target, a larger
// one by a CTA on a bitmap.
constexpr int32_t kWalkMax = 64;

// The n targets of a large cell, at o of the bucket, in id order: ranks from a
// bitmap over the tile (base: its first id), by the whole CTA.
__device__ __forceinline__ void place_large_cell(int32_t o, int32_t n, int32_t base,
                                                 uint32_t* s_bits, int32_t* s_below,
                                                 const int32_t* __restrict__ tmp_id,
                                                 const int32_t* __restrict__ tmp_pos,
                                                 int32_t* __restrict__ fb_id,
                                                 int32_t* __restrict__ fb_pos, int32_t* status) {
  const int tid = threadIdx.x;
  constexpr int kBatch = 4;  // loads in flight per thread
  __syncthreads();
  if (tid < kTileWords) s_bits[tid] = 0;
  __syncthreads();
  for (int32_t i0 = tid; i0 < n; i0 += kBatch * kThreads) {
    int32_t v[kBatch];
#pragma unroll
    for (int q = 0; q < kBatch; ++q)
      v[q] = i0 + q * kThreads < n ? tmp_id[o + i0 + q * kThreads] - base : -1;
#pragma unroll
    for (int q = 0; q < kBatch; ++q) {
      const uint32_t bit = 1u << (v[q] & 31);
      if (v[q] >= 0 && (atomicOr(s_bits + (v[q] >> 5), bit) & bit)) atomicOr(status, kErrTargetDup);
    }
  }
  __syncthreads();
  if (tid < 32) {  // ids below each word: a lane takes four words
    const uint4 w = reinterpret_cast<const uint4*>(s_bits)[tid];
    const int32_t c0 = __popc(w.x), c1 = __popc(w.y), c2 = __popc(w.z);
    const int32_t own = c0 + c1 + c2 + __popc(w.w);
    const int32_t ex = warp_incl_scan(own) - own;
    reinterpret_cast<int4*>(s_below)[tid] = make_int4(ex, ex + c0, ex + c0 + c1, ex + c0 + c1 + c2);
  }
  __syncthreads();
  for (int32_t i0 = tid; i0 < n; i0 += kBatch * kThreads) {
    int32_t v[kBatch], pos[kBatch];
#pragma unroll
    for (int q = 0; q < kBatch; ++q) {
      const int32_t i = i0 + q * kThreads;
      v[q] = i < n ? tmp_id[o + i] - base : -1;
      pos[q] = i < n ? tmp_pos[o + i] : 0;
    }
#pragma unroll
    for (int q = 0; q < kBatch; ++q) {
      if (v[q] < 0) continue;
      const int32_t w = v[q] >> 5;
      const int32_t at = o + s_below[w] + __popc(s_bits[w] & ((1u << (v[q] & 31)) - 1u));
      fb_id[at] = base + v[q];
      fb_pos[at] = pos[q];
    }
  }
}

// Orders each cell's targets by id and flags a target repeated within a
// minibatch.  In a cell of up to kWalkMax targets a thread per slot counts the
// smaller ids: neighbouring slots share a cell, so its ids are read from L1, and
// the work is spread over the whole grid however few cells hold the targets.  (A
// warp per 32 cells, sorting them one after another, took 5 us of a hyperbatch of
// 16 x 1024 targets on 10M nodes, 623 -> 619 us.)  That work grows with the square
// of a cell, so a larger cell is placed by the CTA that holds its first slot.  A
// cell with more entries than a tile has ids repeats one, and is not placed.
// Bucketing of 4 x 65536 consecutive targets: walked 340 us, a warp per 32 cells
// 184, like this 29; 4 x 2M random ones on 2M nodes 9.7, 2.0 and 0.9 ms.  With a
// limit of 32, 64, 128, 256, 512: 8 x 8192 on 100k nodes 31, 31, 33, 35, 41 us,
// 64 x 500 consecutive ones 17, 17, 19, 21, 31, 8 x 1024 on 100k nodes 19, 17, 17,
// 16, 17.
__global__ void __launch_bounds__(kThreads)
targets_place_kernel(const int32_t* __restrict__ fcell_off, int64_t total, int64_t capK, int32_t H,
                     TileMap tm, const int32_t* __restrict__ tmp_id,
                     const int32_t* __restrict__ tmp_pos, int32_t* __restrict__ fb_id,
                     int32_t* __restrict__ fb_pos, int32_t* status) {
  grid_dep_wait();
  if (cta_failed(status)) return;
  __shared__ __align__(16) uint32_t s_bits[kTileWords];
  __shared__ __align__(16) int32_t s_below[kTileWords];
  __shared__ int32_t s_large;
  __shared__ int3 s_cell[kThreads / kWalkMax + 1];  // large cells that start in the chunk
  const int tid = threadIdx.x;
  const int64_t stride = (int64_t)gridDim.x * kThreads;
  for (int64_t s0 = (int64_t)blockIdx.x * kThreads; s0 < total; s0 += stride) {
    const int64_t s = s0 + tid;
    bool starts = false;  // the slot is the first of a large cell
    int3 large = make_int3(0, 0, 0);
    if (s < total) {
      const int32_t v = tmp_id[s];
      const int32_t pos = tmp_pos[s];
      const int32_t t = tile_of(tm, v);
      const int64_t cell = (int64_t)t * H + (uint32_t)pos / (uint32_t)capK;
      const int32_t o = fcell_off[cell], e = fcell_off[cell + 1];
      if (e - o > kTileSpan) {
        atomicOr(status, kErrTargetDup);
      } else if (e - o > kWalkMax) {
        starts = s == o;
        large = make_int3(o, e - o, __ldg(tm.tile_first + t));
      } else {
        int32_t smaller = 0, same = 0;
#pragma unroll 4
        for (int32_t q = o; q < e; ++q) {
          const int32_t u = tmp_id[q];
          smaller += u < v;
          same += u == v;
        }
        if (same > 1) atomicOr(status, kErrTargetDup);
        fb_id[o + smaller] = v;
        fb_pos[o + smaller] = pos;
      }
    }
    if (!__syncthreads_or(starts)) continue;
    if (tid == 0) s_large = 0;
    __syncthreads();
    if (starts) s_cell[atomicAdd(&s_large, 1)] = large;
    __syncthreads();
    const int32_t n = s_large;
    for (int32_t c = 0; c < n; ++c)
      place_large_cell(s_cell[c].x, s_cell[c].y, s_cell[c].z, s_bits, s_below, tmp_id, tmp_pos,
                       fb_id, fb_pos, status);
    __syncthreads();  // the list is rewritten by the next chunk
  }
}

// All of it in one CTA, for few targets on few cells (a request): a thread per
// target, the slots in shared memory, barriers in place of three launches (1 x 16
// targets: 104 -> 99 us a hyperbatch).  With a target and 32 cells per thread the
// CTA's own rounds stay as short as one of those launches; eight targets a thread
// gained nothing at 1024 targets.
constexpr int kFewTargets = kThreads;
constexpr int kFewItems = 32;  // cells per thread, their counts loaded together
constexpr int64_t kFewCells = (int64_t)kThreads * kFewItems;

// Exclusive scan of n <= kFewCells counts into out (n + 1 entries) by one CTA;
// the counts are left zero.  in and out are 16-byte aligned.
__device__ __forceinline__ void few_cells_scan(int32_t* in, int32_t* out, int32_t n) {
  __shared__ int32_t s_w[kWarps];
  const int lane = lane_id(), warp = threadIdx.x >> 5;
  const int32_t i0 = (int32_t)threadIdx.x * kFewItems;
  int32_t v[kFewItems], mine = 0;
#pragma unroll
  for (int q = 0; q < kFewItems / 4; ++q) {
    const int32_t i = i0 + 4 * q;
    int4 x = make_int4(0, 0, 0, 0);
    if (i + 4 <= n) {
      x = __ldcg(reinterpret_cast<const int4*>(in + i));  // counted by atomics at L2
    } else {
      if (i < n) x.x = __ldcg(in + i);
      if (i + 1 < n) x.y = __ldcg(in + i + 1);
      if (i + 2 < n) x.z = __ldcg(in + i + 2);
    }
    v[4 * q] = x.x;
    v[4 * q + 1] = x.y;
    v[4 * q + 2] = x.z;
    v[4 * q + 3] = x.w;
  }
#pragma unroll
  for (int k = 0; k < kFewItems; ++k) mine += v[k];
  const int32_t incl = warp_incl_scan(mine);
  if (lane == 31) s_w[warp] = incl;
  __syncthreads();
  int32_t run = incl - mine;
  for (int q = 0; q < warp; ++q) run += s_w[q];
#pragma unroll
  for (int k = 0; k < kFewItems; ++k) {
    if (i0 + k < n) {
      out[i0 + k] = run;
      in[i0 + k] = 0;
    }
    run += v[k];
    if (i0 + k == n - 1) out[n] = run;
  }
}

__global__ void __launch_bounds__(kThreads)
targets_few_kernel(const int32_t* __restrict__ nodes, int64_t capK, int32_t H, int32_t B,
                   int32_t N, TileMap tm, int32_t* __restrict__ fcnt,
                   int32_t* __restrict__ fcell_off, int32_t cells, int32_t* __restrict__ fb_id,
                   int32_t* __restrict__ fb_pos, int32_t* status) {
  grid_dep_wait();
  __shared__ int32_t s_id[kFewTargets];
  const int32_t i = (int32_t)threadIdx.x;
  const int32_t j = i / B;
  const int32_t pos = (int32_t)(j * capK + (i - j * B));
  const bool has = i < H * B;
  const int32_t v = has ? nodes[pos] : 0;
  const bool bad = v < 0 || v >= N;
  if (bad) atomicOr(status, kErrTargetRange);
  const int32_t cell = has && !bad ? tile_of(tm, v) * H + j : -1;
  const int32_t rank = cell >= 0 ? atomicAdd(fcnt + cell, 1) : 0;
  __threadfence();
  const bool any_bad = __syncthreads_or(bad);
  few_cells_scan(fcnt, fcell_off, cells);  // whatever the ids: the counters are cleared
  if (any_bad) return;
  __syncthreads();
  const int32_t o = cell >= 0 ? fcell_off[cell] : 0, e = cell >= 0 ? fcell_off[cell + 1] : 0;
  if (cell >= 0) s_id[o + rank] = v;
  __syncthreads();
  if (cell < 0) return;
  int32_t smaller = 0, same = 0;
  for (int32_t q = o; q < e; ++q) {
    smaller += s_id[q] < v;
    same += s_id[q] == v;
  }
  if (same > 1) atomicOr(status, kErrTargetDup);
  fb_id[o + smaller] = v;
  fb_pos[o + smaller] = pos;
}

// ---- sampling --------------------------------------------------------------------

// Edge offsets of one hop: indptr of every minibatch's dst list, the exclusive
// scan of min(deg(nodes[i]), k) with the total at the end (also ecnt[j]).
//
// One pass (Merrill & Garland's decoupled look-back, 2016, per minibatch): a
// CTA takes the next (tile of kIndptrTile dst rows, minibatch) pair from a
// counter, tile-major, reads the rows' degrees, publishes the tile's sum and
// walks back over its minibatch's earlier tiles until it meets an inclusive
// prefix.  Pairs are taken in order, so a CTA waits only on pairs of CTAs that
// are already running, and every wait is bounded.  Reading the degrees here in
// dst order replaces a kernel that counted in bucket order, its scattered
// counts, and the two passes over them: 16 x 1024 targets at [15, 10, 5] on 10M
// nodes 653 -> 638 us a hyperbatch, 1 x 1024 272 -> 256 us.
//
// Scratch (uint64, zero on entry; the hop's scatter clears it): [0] the
// counter, [1 + j * tiles + t] flag of minibatch j's tile t = state << 62 |
// value, state 1 = the tile's sum, 2 = the inclusive prefix through it.
constexpr int kIndptrItems = 8;  // rows per thread; hop 3 of 64 x 1024 targets on 40M nodes
                                 // with 4, 8, 16: 31, 27, 35 us; 16 x 1024 on 10M: 16, 18, 26
constexpr int kIndptrTile = kThreads * kIndptrItems;
constexpr unsigned long long kFlagAgg = 1ull << 62;
constexpr unsigned long long kFlagInc = 2ull << 62;
constexpr unsigned long long kFlagVal = (1ull << 62) - 1;
constexpr int kIndptrSpinLimit = 1 << 20;

struct IndptrArgs {
  const int32_t* nodes;  // minibatch j's dst ids at j * capK
  const int32_t* nsz;    // H: |dst|
  const void* offsets;
  bool off32;
  int64_t capK, cap_prev;
  int32_t H, k, tiles;  // tiles: ceil(cap_prev / kIndptrTile)
  int64_t* indptr;
  int32_t* ecnt;
  unsigned long long* scratch;
  int32_t* status;
};

template <typename OffT>
__global__ void __launch_bounds__(kThreads) sample_indptr_kernel(IndptrArgs a) {
  grid_dep_wait();
  if (cta_failed(a.status)) return;
  __shared__ int32_t s_ticket;
  __shared__ int32_t warp_tot[kWarps];
  __shared__ int64_t s_excl;
  const int tid = threadIdx.x, lane = lane_id(), warp = tid >> 5;
  // pairs up to the longest minibatch's last tile
  int32_t longest = 0;
  for (int32_t j = tid; j < a.H; j += kThreads) longest = max(longest, a.nsz[j]);
  longest = __reduce_max_sync(0xffffffffu, longest);
  if (lane == 0) warp_tot[warp] = longest;
  __syncthreads();
  for (int w = 0; w < kWarps; ++w) longest = max(longest, warp_tot[w]);
  const int32_t pairs = max(1, (longest + kIndptrTile - 1) / kIndptrTile) * a.H;  // < 2^31
  const OffT* off = (const OffT*)a.offsets;
  for (;;) {
    __syncthreads();  // the shared words are rewritten
    if (tid == 0) s_ticket = (int32_t)atomicAdd(a.scratch, 1ull);
    __syncthreads();
    const int32_t ticket = s_ticket;
    if (ticket >= pairs) break;
    const int32_t t = ticket / a.H, j = ticket - t * a.H;
    const int32_t len = a.nsz[j];
    const int32_t begin = t * kIndptrTile;
    if (begin >= len && t > 0) continue;
    unsigned long long* flags = a.scratch + 1 + (int64_t)j * a.tiles;
    // a warp's 256 rows as eight coalesced 32-wide slices
    const int32_t* nodes = a.nodes + (int64_t)j * a.capK;
    const int32_t wbase = begin + warp * (32 * kIndptrItems);
    int32_t v[kIndptrItems], c[kIndptrItems];
#pragma unroll
    for (int q = 0; q < kIndptrItems; ++q) {
      const int32_t i = wbase + 32 * q + lane;
      v[q] = i < len ? nodes[i] : -1;
    }
#pragma unroll
    for (int q = 0; q < kIndptrItems; ++q) {
      c[q] = 0;
      if (v[q] >= 0) {
        const int64_t d = (int64_t)__ldg(off + v[q] + 1) - (int64_t)__ldg(off + v[q]);
        c[q] = (int32_t)(d < a.k ? d : a.k);
      }
    }
    int32_t sum = 0;  // exclusive within the warp, slice by slice (a tile's edges < 2^31)
#pragma unroll
    for (int q = 0; q < kIndptrItems; ++q) {
      const int32_t incl = warp_incl_scan(c[q]);
      c[q] = sum + incl - c[q];
      sum += __shfl_sync(0xffffffffu, incl, 31);
    }
    if (lane == 0) warp_tot[warp] = sum;
    __syncthreads();
    if (warp == 0) {
      const int32_t w = lane < kWarps ? warp_tot[lane] : 0;
      const int32_t wi = warp_incl_scan(w);
      const int64_t agg = __shfl_sync(0xffffffffu, wi, kWarps - 1);
      if (lane < kWarps) warp_tot[lane] = wi - w;
      int64_t excl = 0;
      if (t > 0) {
        if (lane == 0) atomicExch(flags + t, kFlagAgg | (unsigned long long)agg);
        for (int32_t p = t - 1;; p -= 32) {
          const int32_t idx = p - lane;  // lane 0 the nearest predecessor
          unsigned long long f = kFlagInc;  // before tile 0: an inclusive prefix of 0
          if (idx >= 0) {
            f = *(const volatile unsigned long long*)(flags + idx);
            for (int spin = 0; (f >> 62) == 0; ++spin) {
              if (spin == kIndptrSpinLimit) {
                atomicOr(a.status, kErrWaitTimeout);
                f = kFlagInc;
                break;
              }
              __nanosleep(32);
              f = *(const volatile unsigned long long*)(flags + idx);
            }
          }
          const unsigned inc = __ballot_sync(0xffffffffu, (f >> 62) == 2);
          const int stop = inc ? __ffs(inc) - 1 : 31;  // lanes 0 .. stop contribute
          excl += warp_sum(lane <= stop ? (int64_t)(f & kFlagVal) : (int64_t)0);
          if (inc) break;
        }
      }
      if (lane == 0) {
        atomicExch(flags + t, kFlagInc | (unsigned long long)(excl + agg));
        s_excl = excl;
        if (begin + kIndptrTile >= len) {  // the minibatch's last tile
          a.indptr[(int64_t)j * (a.cap_prev + 1) + len] = excl + agg;
          a.ecnt[j] = (int32_t)(excl + agg);
        }
      }
    }
    __syncthreads();
    const int64_t base = s_excl + warp_tot[warp];
    int64_t* indptr = a.indptr + (int64_t)j * (a.cap_prev + 1);
#pragma unroll
    for (int q = 0; q < kIndptrItems; ++q) {
      const int32_t i = wbase + 32 * q + lane;
      if (i < len) indptr[i] = base + c[q];
    }
  }
}

struct FillArgs {
  TileMap tm;
  // frontier entries [fcell_off[cell_lo], fcell_off[cell_hi]) are sampled
  const int32_t* fcell_off;
  int64_t cell_lo, cell_hi;
  // streamed topology: edge lists of resident physical blocks in the graph
  // buffer (slot * epb edges each); blk_slot[b] < 0 means not resident
  const int32_t* tile_adj_block;
  const int32_t* blk_slot;
  const int64_t* blk_e0;
  const int32_t* gbuf;
  int64_t epb, hdr, bb;
  int32_t H;
  int32_t* scnt;   // T*H per-cell counters of sampled ids (zero on entry)
  int32_t* scell;  // per edge: its (tile, minibatch) cell
  int32_t* srank;  // per edge: its rank within the cell
  const int32_t* fb_id;
  const int32_t* fb_pos;
  const void* offsets;
  bool off32;
  const int64_t* indptr;
  const int32_t* indices;
  int32_t* nbr;
  int64_t capK, cap_prev, ecap;
  int32_t k, hop;
  const uint64_t* key;  // device: {seed, first minibatch id}
  int32_t* status;
  bool packed;        // record rank << 12 | tile-local id in nbr, no srank (the dedup's
                      // sampled bucket is packed)
  int32_t* hset;      // fanouts above kWideMax: per-warp hash sets of chosen positions
  int32_t hset_log2;  // each of 2^hset_log2 entries
};

// The sampling key, read from device memory once per thread, so that one
// captured launch sequence serves every seed and minibatch id.
struct Key {
  uint32_t lo, hi;
  uint64_t gid0;
};

__device__ __forceinline__ Key load_key(const uint64_t* key) {
  const uint64_t seed = __ldg(key);
  return Key{(uint32_t)seed, (uint32_t)(seed >> 32), __ldg(key + 1)};
}

// First edge and degree of node v.  Entries are walked in bucket order, so
// neighbouring lanes' offsets share cache lines.
__device__ __forceinline__ longlong2 first_and_degree(const FillArgs& a, int32_t v) {
  int64_t lo, hi;
  if (a.off32) {
    const int32_t* off = (const int32_t*)a.offsets + v;
    lo = __ldg(off);
    hi = __ldg(off + 1);
  } else {
    const int64_t* off = (const int64_t*)a.offsets + v;
    lo = __ldg(off);
    hi = __ldg(off + 1);
  }
  return make_longlong2(lo, hi - lo);
}

// Where the sampler reads neighbour entries.
enum EdgeSrc : int {
  kEdgesInPlace = 0,  // a.indices (HBM, or the device view of pinned host memory)
  kEdgesBuffer = 1,   // the graph buffer: every needed block is resident
  kEdgesCached = 2,   // the topology cache where the block is cached, else in place
};

// Neighbour at position pos of node v (edges off_v .. off_v + deg).  In the
// graph buffer or the topology cache the edge sits in the slot of its
// physical block: v's first block, plus, for an object larger than a block,
// the block its byte offset (after the header) falls in.
template <int kSrc>
__device__ __forceinline__ int32_t edge_at(const FillArgs& a, int32_t v, int64_t off_v,
                                           int64_t deg, int64_t pos) {
  if (kSrc == kEdgesInPlace) return __ldg(a.indices + off_v + pos);
  int64_t b = __ldg(a.tile_adj_block + tile_of(a.tm, v));
  if (a.hdr + 4 * deg > a.bb) b += (a.hdr + 4 * pos) / a.bb;
  const int32_t slot = __ldg(a.blk_slot + b);
  if (slot < 0) {
    if (kSrc == kEdgesCached) return __ldg(a.indices + off_v + pos);
    atomicOr(a.status, kErrInternal);  // cannot happen: the host made every needed block resident
    return 0;
  }
  return __ldg(a.gbuf + (int64_t)slot * a.epb + (off_v + pos - __ldg(a.blk_e0 + b)));
}

__device__ __forceinline__ int64_t draw(const FillArgs& a, const Key& key, int32_t v, int32_t s,
                                        uint64_t gid, int64_t J) {
  const uint4 x = philox4x32_10(
      make_uint4((uint32_t)v, ((uint32_t)a.hop << 24) | (uint32_t)s, (uint32_t)gid,
                 (uint32_t)(gid >> 32)),
      make_uint2(key.lo, key.hi));
  const uint64_t r = ((uint64_t)x.y << 32) | (uint64_t)x.x;
  return (int64_t)__umul64hi(r, (uint64_t)(J + 1));
}

// Records sampled edge e = (j, eidx) with neighbour u: its id, its
// (tile, minibatch) cell and its rank within the cell (one atomic per distinct
// cell of the warp), so the bucketing scatter after the scan needs no atomics.
// Called by all 32 lanes; lanes without an edge pass has = false.  Cell
// indices fit 31 bits (T * H < 2^31).
__device__ __forceinline__ void emit_edges(const FillArgs& a, bool has, int32_t u, uint32_t j,
                                           int64_t eidx) {
  const int32_t t = tile_of(a.tm, has ? u : 0);
  const uint32_t cell = (uint32_t)t * (uint32_t)a.H + j;
  // the id, or with a packed sampled bucket its tile-local id
  const int32_t val = a.packed ? u - __ldg(a.tm.tile_first + t) : u;
  const unsigned peers = __match_any_sync(0xffffffffu, has ? cell : 0xffffffffu);
  const int lane = lane_id();
  const int leader = __ffs(peers) - 1;
  int32_t old = 0;
  if (has && lane == leader) old = atomicAdd(a.scnt + cell, __popc(peers));
  old = __shfl_sync(0xffffffffu, old, leader);
  if (has) {
    const int64_t at = (int64_t)j * a.ecap + eidx;
    const int32_t rank = old + __popc(peers & ((1u << lane) - 1u));
    a.scell[at] = (int32_t)cell;
    if (a.packed) {  // rank < ecap <= 2^20 beside the 12-bit tile-local id
      a.nbr[at] = (rank << 12) | val;
    } else {
      a.nbr[at] = val;
      a.srank[at] = rank;
    }
  }
}

// k <= 32: k lanes per frontier node (lane s draws slot s), 32 / k nodes per
// warp round; the lanes past them (32 mod k) idle.  The round runs without
// divergent branches: every lane draws (a node of degree <= k takes its
// first d edges instead) and the collision shuffles span the whole warp.
template <int kSrc>
__global__ void __launch_bounds__(kThreads, 8) sample_fill_kernel(FillArgs a) {
  grid_dep_wait();
  if (failed(a.status)) return;
  const Key key = load_key(a.key);
  const int64_t E0 = a.fcell_off[a.cell_lo], E1 = a.fcell_off[a.cell_hi];
  const int k = a.k;
  const int groups = 32 / k;
  const int lane = lane_id();
  const int sub = lane / k, s = lane - sub * k;
  const int g0 = sub * k;  // the group's first lane (>= 32 - k for idle lanes)
  const bool member = sub < groups;
  const uint32_t capk32 = (uint32_t)a.capK;
  const int64_t warp0 = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t e0 = E0 + warp0 * groups; e0 < E1; e0 += nwarps * groups) {
    const int64_t i = e0 + sub;
    const bool live = member && i < E1;
    int32_t v = 0;
    uint32_t g = 0;
    longlong2 bd = make_longlong2(0, 0);
    if (live) {
      v = a.fb_id[i];
      g = (uint32_t)a.fb_pos[i];
      bd = first_and_degree(a, v);
    }
    const int64_t base = bd.x, d = bd.y;
    const uint32_t j = g / capk32;
    const uint32_t pos = g - j * capk32;
    int64_t eidx = s;
    if (live) eidx += a.indptr[j * (a.cap_prev + 1) + pos];
    // Floyd's algorithm: slot s draws t in [0, J], J = d - k + s, and takes J
    // when an earlier slot of the node holds t
    const int64_t J = d - k + s;
    const int64_t t = draw(a, key, v, s, key.gid0 + j, J);
    bool collided = false;
    if (__any_sync(0xffffffffu, d > (int64_t)0xffffffffu)) {  // positions past 32 bits
      for (int q = 0; q < k; ++q) {
        const int64_t cq = __shfl_sync(0xffffffffu, collided ? J : t, g0 + q);
        if (s > q && t == cq) collided = true;
      }
    } else {
      const uint32_t t32 = (uint32_t)t, J32 = (uint32_t)J;
      for (int q = 0; q < k; ++q) {
        const uint32_t cq = __shfl_sync(0xffffffffu, collided ? J32 : t32, g0 + q);
        if (s > q && t32 == cq) collided = true;
      }
    }
    const bool small = d <= k;
    const bool has = live && (!small || s < d);
    int32_t u = 0;
    if (has) u = edge_at<kSrc>(a, v, base, d, small ? (int64_t)s : collided ? J : t);
    emit_edges(a, has, u, j, eidx);
  }
}

// One warp per frontier node for fanouts above 32: slots are drawn 32 at a
// time; each candidate is checked against the choices of earlier chunks (kept
// in shared memory) and then resolved within its chunk by shuffles.
template <int kSrc>
__global__ void __launch_bounds__(kThreads) sample_fill_wide_kernel(FillArgs a) {
  grid_dep_wait();
  if (failed(a.status)) return;
  __shared__ int32_t chosen_s[kWarps][kWideMax];
  const int warp = threadIdx.x >> 5, lane = lane_id();
  int32_t* chosen = chosen_s[warp];
  const Key key = load_key(a.key);
  const int64_t E0 = a.fcell_off[a.cell_lo], E1 = a.fcell_off[a.cell_hi];
  const uint32_t capk32 = (uint32_t)a.capK;
  const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t i = E0 + ((blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5); i < E1;
       i += nwarps) {
    const int32_t v = a.fb_id[i];
    const uint32_t g = (uint32_t)a.fb_pos[i];
    const uint32_t j = g / capk32;
    const uint32_t pos = g - j * capk32;
    const longlong2 bd = first_and_degree(a, v);
    const int64_t base = bd.x, d = bd.y;
    const int64_t ebase = a.indptr[j * (a.cap_prev + 1) + pos];
    if (d <= a.k) {
      for (int64_t q0 = 0; q0 < d; q0 += 32) {
        const int64_t q = q0 + lane;
        const bool has = q < d;
        emit_edges(a, has, has ? edge_at<kSrc>(a, v, base, d, q) : 0, j, ebase + q);
      }
      continue;
    }
    for (int c0 = 0; c0 < a.k; c0 += 32) {
      const int s = c0 + lane;
      const bool valid = s < a.k;
      const int64_t J = d - a.k + s;
      const int64_t t = valid ? draw(a, key, v, s, key.gid0 + j, J) : -1;
      bool collided = false;
      for (int q = 0; q < c0; ++q) collided |= (chosen[q] == t);
      const int m = min(32, a.k - c0);
      for (int q = 0; q < m; ++q) {
        const int64_t mine = collided ? J : t;
        const int64_t cq = __shfl_sync(0xffffffffu, mine, q);
        if (lane > q && t == cq) collided = true;
      }
      const int64_t c = collided ? J : t;
      if (valid) chosen[s] = (int32_t)c;
      emit_edges(a, valid, valid ? edge_at<kSrc>(a, v, base, d, c) : 0, j, ebase + s);
      __syncwarp();
    }
  }
}

// ---- fanouts above kWideMax -----------------------------------------------------
//
// One warp per frontier node, slots drawn 32 at a time as in the wide sampler;
// the positions chosen by earlier chunks live in the warp's own open-addressing
// hash set in global memory (2^hset_log2 >= 2k entries, so it is at most half
// full and every probe sequence ends at an empty entry within the table),
// cleared for each node.  Lookups bypass L1 (__ldcg): the set's entries are
// written by the warp's atomics at L2.
constexpr int32_t kHsetEmpty = -1;

__device__ __forceinline__ uint32_t hset_slot(int32_t key, uint32_t mask) {
  return ((uint32_t)key * 0x9E3779B1u) & mask;  // Fibonacci hashing, low bits
}

__device__ __forceinline__ bool hset_contains(const int32_t* T, uint32_t mask, int32_t key) {
  uint32_t h = hset_slot(key, mask);
  for (uint32_t probe = 0; probe <= mask; ++probe) {
    const int32_t v = __ldcg(T + h);
    if (v == key) return true;
    if (v == kHsetEmpty) return false;
    h = (h + 1u) & mask;
  }
  return false;
}

// Inserts key (distinct from the keys other lanes insert at the same time).
__device__ __forceinline__ void hset_insert(int32_t* T, uint32_t mask, int32_t key) {
  uint32_t h = hset_slot(key, mask);
  for (uint32_t probe = 0; probe <= mask; ++probe) {
    const int32_t old = atomicCAS(T + h, kHsetEmpty, key);
    if (old == kHsetEmpty || old == key) return;
    h = (h + 1u) & mask;
  }
}

template <int kSrc>
__global__ void __launch_bounds__(kThreads) sample_fill_huge_kernel(FillArgs a) {
  grid_dep_wait();
  if (failed(a.status)) return;
  const int lane = lane_id();
  const Key key = load_key(a.key);
  const int64_t E0 = a.fcell_off[a.cell_lo], E1 = a.fcell_off[a.cell_hi];
  const uint32_t capk32 = (uint32_t)a.capK;
  const int64_t gw = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  const uint32_t mask = (1u << a.hset_log2) - 1u;
  int32_t* T = a.hset + (gw << a.hset_log2);
  for (int64_t i = E0 + gw; i < E1; i += nwarps) {
    const int32_t v = a.fb_id[i];
    const uint32_t g = (uint32_t)a.fb_pos[i];
    const uint32_t j = g / capk32;
    const uint32_t pos = g - j * capk32;
    const longlong2 bd = first_and_degree(a, v);
    const int64_t base = bd.x, d = bd.y;
    const int64_t ebase = a.indptr[j * (a.cap_prev + 1) + pos];
    if (d <= a.k) {
      for (int64_t q0 = 0; q0 < d; q0 += 32) {
        const int64_t q = q0 + lane;
        const bool has = q < d;
        emit_edges(a, has, has ? edge_at<kSrc>(a, v, base, d, q) : 0, j, ebase + q);
      }
      continue;
    }
    for (uint32_t w = (uint32_t)lane; w <= (mask >> 2); w += 32)
      reinterpret_cast<int4*>(T)[w] = make_int4(kHsetEmpty, kHsetEmpty, kHsetEmpty, kHsetEmpty);
    __syncwarp();
    for (int c0 = 0; c0 < a.k; c0 += 32) {
      const int s = c0 + lane;
      const bool valid = s < a.k;
      const int64_t J = d - a.k + s;
      const int64_t t = valid ? draw(a, key, v, s, key.gid0 + j, J) : -1;
      bool collided = valid && hset_contains(T, mask, (int32_t)t);
      const int m = min(32, a.k - c0);
      for (int q = 0; q < m; ++q) {
        const int64_t mine = collided ? J : t;
        const int64_t cq = __shfl_sync(0xffffffffu, mine, q);
        if (lane > q && t == cq) collided = true;
      }
      const int64_t c = collided ? J : t;
      if (valid) hset_insert(T, mask, (int32_t)c);
      emit_edges(a, valid, valid ? edge_at<kSrc>(a, v, base, d, c) : 0, j, ebase + s);
      __syncwarp();  // the chunk's inserts are seen by the next chunk's lookups
    }
    __syncwarp();  // every lookup of this node is done before the next clear
  }
}

}  // namespace

int64_t huge_fanout_tables(int32_t k, int num_sms, int32_t* log2, int32_t* grid) {
  *log2 = 0;
  *grid = 0;
  if (k <= kWideMax) return 0;
  int32_t l = 2;
  while ((1 << l) < 2 * k) ++l;
  int g = resident_grid((const void*)sample_fill_huge_kernel<kEdgesInPlace>, kThreads, num_sms);
  const int64_t budget_entries = (int64_t)1 << 28;  // 1 GiB of tables at most
  const int64_t max_warps = budget_entries >> l;
  if ((int64_t)g * kWarps > max_warps) g = (int)(max_warps / kWarps);
  if (g < 1) g = 1;
  *log2 = l;
  *grid = g;
  return ((int64_t)g * kWarps) << l;
}

cudaError_t launch_bucket_targets(int32_t* nodes, int64_t capK, int32_t H, int32_t B, int32_t N,
                                  const int32_t* tile_first, const int32_t* chunk_tile, int32_t T,
                                  int32_t* fcnt, int32_t* fcell_off, int32_t* tmp_id,
                                  int32_t* tmp_pos, int32_t* fb_id, int32_t* fb_pos,
                                  uint64_t* flat_scratch, int32_t* status, int num_sms,
                                  cudaStream_t st) {
  const TileMap tm{tile_first, chunk_tile, T};
  const int64_t ncells = (int64_t)T * H;
  const int64_t total = (int64_t)H * B;
  if (total <= kFewTargets && ncells <= kFewCells) {
    targets_few_kernel<<<1, kThreads, 0, st>>>(nodes, capK, H, B, N, tm, fcnt, fcell_off,
                                               (int32_t)ncells, fb_id, fb_pos, status);
    return cudaGetLastError();
  }
  auto grid = [&](const void* kernel) {  // a thread per target
    return fitted_grid(kernel, kThreads, num_sms, (total + kThreads - 1) / kThreads);
  };
  int32_t* rank = fb_id;  // free until the bucket is written
  targets_count_kernel<<<grid((const void*)targets_count_kernel), kThreads, 0, st>>>(
      nodes, capK, H, B, N, tm, fcnt, rank, status);
  cudaError_t e =
      flat_scan(fcnt, fcell_off, ncells, true, flat_scratch, status, st);
  if (e != cudaSuccess) return e;
  targets_scatter_kernel<<<grid((const void*)targets_scatter_kernel), kThreads, 0, st>>>(
      nodes, capK, H, B, tm, fcell_off, rank, tmp_id, tmp_pos, status);
  targets_place_kernel<<<grid((const void*)targets_place_kernel), kThreads, 0, st>>>(
      fcell_off, total, capK, H, tm, tmp_id, tmp_pos, fb_id, fb_pos, status);
  return cudaGetLastError();
}

int64_t indptr_scratch_elems(int32_t H, int64_t cap_prev) {
  return 1 + H * ((cap_prev + kIndptrTile - 1) / kIndptrTile);
}

cudaError_t launch_sample_indptr(const HopArgs& a, const int32_t* nodes, const int32_t* nsz,
                                 int64_t* indptr, int32_t* ecnt, uint64_t* scratch, int num_sms,
                                 cudaStream_t st) {
  IndptrArgs p;
  p.nodes = nodes;
  p.nsz = nsz;
  p.offsets = a.offsets;
  p.off32 = a.offsets_bits == 32;
  p.capK = a.capK;
  p.cap_prev = a.cap_prev;
  p.H = a.H;
  p.k = a.k;
  p.tiles = (int32_t)((a.cap_prev + kIndptrTile - 1) / kIndptrTile);
  p.indptr = indptr;
  p.ecnt = ecnt;
  p.scratch = reinterpret_cast<unsigned long long*>(scratch);
  p.status = a.status;
  const void* kernel = p.off32 ? (const void*)sample_indptr_kernel<int32_t>
                               : (const void*)sample_indptr_kernel<int64_t>;
  const int grid = fitted_grid(kernel, kThreads, num_sms, (int64_t)p.tiles * a.H);
  if (p.off32)
    sample_indptr_kernel<int32_t><<<grid, kThreads, 0, st>>>(p);
  else
    sample_indptr_kernel<int64_t><<<grid, kThreads, 0, st>>>(p);
  return cudaGetLastError();
}

template <int kSrc>
static void launch_fill_typed(const FillArgs& f, int k, int huge_grid, int num_sms,
                              cudaStream_t st) {
  const int64_t entries = f.H * f.cap_prev;  // at most
  auto grid = [&](const void* kernel, int per_warp) {
    const int64_t per_cta = (int64_t)kWarps * per_warp;
    return fitted_grid(kernel, kThreads, num_sms, (entries + per_cta - 1) / per_cta);
  };
  if (k <= 32)
    sample_fill_kernel<kSrc>
        <<<grid((const void*)sample_fill_kernel<kSrc>, 32 / k), kThreads, 0, st>>>(f);
  else if (k <= kWideMax)
    sample_fill_wide_kernel<kSrc>
        <<<grid((const void*)sample_fill_wide_kernel<kSrc>, 1), kThreads, 0, st>>>(f);
  else
    sample_fill_huge_kernel<kSrc><<<huge_grid, kThreads, 0, st>>>(f);
}

cudaError_t launch_sample_fill(const HopArgs& a, const int32_t* fb_id, const int32_t* fb_pos,
                               const int32_t* fcell_off, const int64_t* indptr, int32_t* nbr,
                               int32_t* scnt, int32_t* scell, int32_t* srank,
                               const FillRange& r, int num_sms, cudaStream_t st) {
  FillArgs f;
  f.tm = TileMap{a.tile_first, a.chunk_tile, a.T};
  f.fcell_off = fcell_off;
  f.cell_lo = r.cell_lo;
  f.cell_hi = r.cell_hi;
  f.tile_adj_block = r.tile_adj_block;
  f.blk_slot = r.blk_slot;
  f.blk_e0 = r.blk_e0;
  f.gbuf = r.gbuf;
  f.epb = r.epb;
  f.hdr = a.offsets_bits / 8;
  f.bb = r.bb;
  f.H = a.H;
  f.scnt = scnt;
  f.scell = scell;
  f.srank = srank;
  f.fb_id = fb_id;
  f.fb_pos = fb_pos;
  f.offsets = a.offsets;
  f.off32 = a.offsets_bits == 32;
  f.indptr = indptr;
  f.indices = a.indices;
  f.nbr = nbr;
  f.capK = a.capK;
  f.cap_prev = a.cap_prev;
  f.ecap = a.ecap;
  f.k = a.k;
  f.hop = a.hop;
  f.key = a.key;
  f.status = a.status;
  f.hset = a.hset;
  f.hset_log2 = a.hset_log2;
  f.packed = a.sb_packed;
  if (a.k > kWideMax && (a.hset == nullptr || a.hset_grid < 1)) return cudaErrorInvalidValue;
  const int src = r.gbuf == nullptr ? kEdgesInPlace : r.in_place_fallback ? kEdgesCached
                                                                            : kEdgesBuffer;
  if (src == kEdgesInPlace)
    launch_fill_typed<kEdgesInPlace>(f, a.k, a.hset_grid, num_sms, st);
  else if (src == kEdgesBuffer)
    launch_fill_typed<kEdgesBuffer>(f, a.k, a.hset_grid, num_sms, st);
  else
    launch_fill_typed<kEdgesCached>(f, a.k, a.hset_grid, num_sms, st);
  return cudaGetLastError();
}

}  // namespace agnes
