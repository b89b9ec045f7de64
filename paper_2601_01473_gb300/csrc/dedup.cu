// dedup.cu -- per-minibatch union / dedup and relabelling of a hop's samples
// (Algorithm 1: N^j_out <- N^j_out u Sample(j, ...), N_in <- N_out).
//
// The sampled ids of every minibatch are bucketed by (tile, minibatch) cell
// (histogram -> scan -> scatter, the bucket matrix of Sec. 3.4 (3)); each
// cell is then resolved once against the same cell of the frontier bucket:
// D = the cell's frontier (dst_h) ids, S = its sampled ids, new = S \ D.
// Tiles ascend in id, so new_h in ascending order is the cells' new ids in
// tile order, and a per-minibatch scan of the cells' new counts over tiles
// places every new node in src_h = dst_h ++ new_h.  Resolving a cell gives,
// with ranks local to the cell, each sampled edge's col and the cell of the
// next hop's frontier bucket (D | new in ascending id); after the scans, a
// fix-up pass and a compaction pass turn the local ranks into final indices.
// The bucket is carried from hop to hop and never rebuilt.  This file holds
// the scatter and the compaction with the fix-up; the cells are resolved in
// dedup_cells.cu.
#include "common.cuh"
#include "compact_index.h"
#include "internal.h"

namespace agnes {

namespace {

constexpr int kThreads = 256;
constexpr int kIlp = 4;  // independent elements per thread in the streaming passes

// Places every sampled edge of minibatch j at soff[cell] + rank (cell and
// rank were recorded while sampling), building the sampled bucket: (id, edge
// index) pairs, or packed 4-byte entries edge index << 12 | tile-local id.  It
// also empties the queue of the cell kernels that follow, clears the indptr
// scan's flags and counts the topology blocks the frontier touches.
__global__ void __launch_bounds__(kThreads)
dedup_scatter_kernel(const int32_t* __restrict__ nbr, const int32_t* __restrict__ ecnt,
                     int64_t ecap, const int32_t* __restrict__ scell,
                     const int32_t* __restrict__ srank, const int32_t* __restrict__ soff,
                     int2* __restrict__ sb, bool packed, int32_t* __restrict__ q_ctl,
                     unsigned long long* __restrict__ clear, int64_t n_clear,
                     const int32_t* __restrict__ fcell_off, int32_t H,
                     const int32_t* __restrict__ run_first_tile, int64_t n_runs,
                     int64_t* __restrict__ touched, const int32_t* status) {
  grid_dep_wait();
  const int64_t i0 =
      ((int64_t)blockIdx.y * gridDim.x + blockIdx.x) * blockDim.x + threadIdx.x;
  const int64_t threads = (int64_t)gridDim.x * gridDim.y * blockDim.x;
  // whatever the status: the next hop or hyperbatch relies on it
  for (int64_t i = i0; i < n_clear; i += threads) clear[i] = 0;
  if (i0 < 2) q_ctl[i0] = 0;
  if (failed(status)) return;
  count_touched(i0, threads, fcell_off, H, run_first_tile, n_runs, touched);
  const int32_t j = blockIdx.y;
  const int64_t E = ecnt[j];
  const int64_t o = (int64_t)j * ecap;
  for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < E;
       e += (int64_t)gridDim.x * blockDim.x) {
    if (packed) {  // nbr holds rank << 12 | tile-local id; e < 2^20
      const uint32_t v = (uint32_t)nbr[o + e];
      reinterpret_cast<uint32_t*>(sb)[soff[scell[o + e]] + (v >> 12)] =
          ((uint32_t)e << 12) | (v & 0xfffu);
    } else {
      sb[soff[scell[o + e]] + srank[o + e]] = make_int2(nbr[o + e], (int32_t)e);
    }
  }
}

constexpr int kCompactOversplit = 2;  // the compaction's (group, slice) items per resident CTA
constexpr int kGroupCells = kCellThreads;

// ---- compaction and fix-up (after the scans) --------------------------------------

struct CompactArgs {
  int64_t ncells;
  int32_t slices;  // CTAs per group of kGroupCells cells
  int32_t H;
  int64_t capK;
  const int32_t* fb_id;
  const int32_t* fb_pos;
  const int32_t* fcell_off;
  const int32_t* soff;
  const int2* tmp;
  const int32_t* nfcell_off;
  const int32_t* newbase;
  const int32_t* nsz_prev;
  const int32_t* noutbase;   // sampled frontier: rows are positions among the distinct samples
  bool sampled;
  int32_t* nfb_id;
  int32_t* nfb_pos;
  int32_t* nodes;
  // the col fix-up: H x ecap edges, ecnt[j] of minibatch j's, fix_ctas CTAs each
  int32_t* col;
  const int32_t* ecnt;
  int64_t ecap;
  const int32_t* scell;
  int32_t fix_ctas;
  // the last hop's count of touched feature blocks (n_feat_blocks 0: none)
  const int32_t* fblock_first_tile;
  int64_t n_feat_blocks;
  int64_t* feat_touched;
  const int32_t* status;
};

// col[e] = -(1 + r) becomes the new node's index in src_h:
// |dst_h| + (new ids of the minibatch in earlier tiles) + r.  kIlp edges per
// thread: their base loads in flight together.
__device__ __forceinline__ void fix_col(const CompactArgs& a, int32_t j, int32_t part) {
  const int64_t E = a.ecnt[j];
  int32_t* col = a.col + (int64_t)j * a.ecap;
  const int32_t* scell = a.scell + (int64_t)j * a.ecap;
  const int32_t base = a.nsz_prev[j];
  const int64_t stride = (int64_t)a.fix_ctas * kCellThreads;
  for (int64_t e0 = (int64_t)part * kCellThreads + threadIdx.x; e0 < E; e0 += kIlp * stride) {
    int32_t v[kIlp], cell[kIlp], nb[kIlp];
#pragma unroll
    for (int k = 0; k < kIlp; ++k) {
      const int64_t e = e0 + k * stride;
      v[k] = e < E ? col[e] : 0;
      cell[k] = e < E ? scell[e] : 0;
    }
#pragma unroll
    for (int k = 0; k < kIlp; ++k) nb[k] = v[k] < 0 ? a.newbase[cell[k]] : 0;
#pragma unroll
    for (int k = 0; k < kIlp; ++k)
      if (v[k] < 0) col[e0 + k * stride] = base + nb[k] + (-1 - v[k]);
  }
}

// Writes the next frontier bucket in cell order: a cell without samples is
// copied from the current bucket, any other from its tmp entries, where a new
// node (x = -(1 + r)) gets its output row j * capK + |dst_h| + newbase + r and
// its id is appended to the minibatch's node list.  A group of kGroupCells
// cells is shared by `slices` CTAs, each taking every slices-th round of its
// entries: small graphs have few groups with many entries each, and the
// entries' loads are latency-bound, so they need every SM (8 minibatches of
// 500 at [25, 10] on 250k nodes: 446 -> 349 us a hyperbatch; two items per
// resident CTA, where four cost 3% and eight 5% on 10M nodes).
// The col fix-up needs the same scans and nothing else, so the CTAs take it on
// afterwards in the same launch.
__global__ void __launch_bounds__(kCellThreads) dedup_compact_kernel(CompactArgs a) {
  grid_dep_wait();
  if (failed(a.status)) return;
  __shared__ int32_t s_nfo[kGroupCells + 1];
  __shared__ int64_t s_src[kGroupCells];   // the cell's first entry in fb, or ~ that in tmp
  __shared__ int32_t s_row[kGroupCells];   // j * capK + |dst_h| + newbase
  const int tid = threadIdx.x;
  const int64_t ngroups = (a.ncells + kGroupCells - 1) / kGroupCells;
  const int64_t nitems = ngroups * a.slices;
  for (int64_t item = blockIdx.x; item < nitems; item += gridDim.x) {
    const int64_t grp = item / a.slices;
    const int32_t slice = (int32_t)(item - grp * a.slices);
    const int64_t c0 = grp * kGroupCells;
    const int64_t cell = c0 + tid;
    const int64_t last = min(a.ncells, c0 + kGroupCells);
    if (cell < a.ncells) {
      const int32_t fo = a.fcell_off[cell];
      const int32_t so = a.soff[cell];
      const int32_t sn = a.soff[cell + 1] - so;
      const int32_t j = (int32_t)((uint32_t)cell % (uint32_t)a.H);
      s_nfo[tid] = a.nfcell_off[cell];
      s_src[tid] = sn == 0 && !a.sampled ? (int64_t)fo : ~tmp_base(fo, so);
      s_row[tid] = (int32_t)((int64_t)j * a.capK +
                             (a.sampled ? a.noutbase[cell] : a.nsz_prev[j] + a.newbase[cell]));
    }
    if (tid == 0) s_nfo[last - c0] = a.nfcell_off[last];
    __syncthreads();
    const int32_t k0 = s_nfo[0];
    const uint32_t k1 = (uint32_t)s_nfo[last - c0];
    // kCompactIlp entries per thread and round: their loads in flight before the stores
    for (uint32_t kb = compact_first(k0, slice, tid); kb < k1; kb = compact_next(kb, a.slices)) {
      int32_t cl[kCompactIlp], r[kCompactIlp], id[kCompactIlp], pos[kCompactIlp];
      bool in[kCompactIlp];
#pragma unroll
      for (int u = 0; u < kCompactIlp; ++u) {
        const uint32_t k = kb + u * kCellThreads;
        in[u] = k < k1;
        int32_t lo = 0, hi = (int32_t)(last - c0);  // last cell with nfo <= k
        while (hi - lo > 1) {
          const int32_t mid = (lo + hi) >> 1;
          if ((uint32_t)s_nfo[mid] <= k) lo = mid; else hi = mid;
        }
        cl[u] = lo;
        r[u] = (int32_t)(k - (uint32_t)s_nfo[lo]);
        id[u] = 0;
        pos[u] = 0;
        if (in[u]) {
          const int64_t src = s_src[lo];
          if (src >= 0) {
            id[u] = a.fb_id[src + r[u]];
            pos[u] = a.fb_pos[src + r[u]];
          } else {
            const int2 e = a.tmp[~src + r[u]];
            id[u] = e.x;
            pos[u] = e.y;
          }
        }
      }
#pragma unroll
      for (int u = 0; u < kCompactIlp; ++u) {
        if (!in[u]) continue;
        const uint32_t k = kb + u * kCellThreads;
        if (s_src[cl[u]] < 0) {
          if (a.sampled) {
            pos[u] = s_row[cl[u]] + r[u];
            a.nodes[pos[u]] = id[u];
          } else if (pos[u] < 0) {
            pos[u] = s_row[cl[u]] + (-1 - pos[u]);
            a.nodes[pos[u]] = id[u];
          }
        }
        a.nfb_id[k] = id[u];
        a.nfb_pos[k] = pos[u];
      }
    }
    __syncthreads();
  }
  const int64_t nfix = (int64_t)a.H * a.fix_ctas;
  for (int64_t f = blockIdx.x; f < nfix; f += gridDim.x) {
    const int32_t j = (int32_t)(f / a.fix_ctas);
    fix_col(a, j, (int32_t)(f - (int64_t)j * a.fix_ctas));
  }
  if (a.n_feat_blocks > 0)
    count_touched(blockIdx.x * (int64_t)kCellThreads + tid, (int64_t)gridDim.x * kCellThreads,
                  a.nfcell_off, a.H, a.fblock_first_tile, a.n_feat_blocks, a.feat_touched);
}

}  // namespace

cudaError_t launch_dedup(const HopArgs& a, const DedupBufs& d, int num_sms, cudaStream_t st) {
  const int64_t ncells = (int64_t)a.T * a.H;
  // CTAs per minibatch: eight per SM in all, no more than its edges fill
  const int64_t gx = (num_sms * 8 + a.H - 1) / a.H, fill = (a.ecap + kThreads - 1) / kThreads;
  const dim3 egrid((unsigned)(gx < fill ? gx : fill), (unsigned)a.H);
  cudaError_t e =
      flat_scan(d.scnt, d.soff, ncells, true, d.flat_scratch, a.status, st);
  if (e != cudaSuccess) return e;
  dedup_scatter_kernel<<<egrid, kThreads, 0, st>>>(d.nbr, d.ecnt, a.ecap, d.scell, d.srank,
                                                   d.soff, d.sb, a.sb_packed, d.q_ctl,
                                                   reinterpret_cast<unsigned long long*>(
                                                       d.indptr_scratch),
                                                   indptr_scratch_elems(a.H, a.cap_prev),
                                                   d.fcell_off, a.H, d.run_first_tile, d.n_runs,
                                                   d.touched, a.status);

  e = launch_dedup_cells(a, d, num_sms, st);  // dedup_cells.cu
  if (e != cudaSuccess) return e;
  // per-minibatch offsets of the new ids: scan down the tiles of the
  // tile-major [T x H] count matrix; totals give the next frontier sizes
  // |src_h| = |dst_h| + new ids; the next frontier is src_h, or (sampled
  // frontier) the distinct sampled ids, numbered by their own column scan.
  const ColumnScan scans[2] = {
      {d.newcnt, d.newbase, d.nsz_prev, {d.srcsz, d.frontier_sampled ? nullptr : d.nsz_next}},
      {d.nfcnt, d.noutbase, nullptr, {d.nsz_next, nullptr}}};
  e = cell_scans(a.T, a.H, d.nfcnt, d.nfcell_off, d.flat_scratch, scans,
                 d.frontier_sampled ? 2 : 1, d.cols_scratch, a.status, st);
  if (e != cudaSuccess) return e;

  CompactArgs k;
  k.ncells = ncells;
  k.H = a.H;
  k.capK = a.capK;
  k.fb_id = d.fb_id;
  k.fb_pos = d.fb_pos;
  k.fcell_off = d.fcell_off;
  k.soff = d.soff;
  k.tmp = d.tmp;
  k.nfcell_off = d.nfcell_off;
  k.newbase = d.newbase;
  k.nsz_prev = d.nsz_prev;
  k.noutbase = d.noutbase;
  k.sampled = d.frontier_sampled;
  k.nfb_id = d.nfb_id;
  k.nfb_pos = d.nfb_pos;
  k.nodes = d.nodes;
  k.col = d.col;
  k.ecnt = d.ecnt;
  k.ecap = a.ecap;
  k.scell = d.scell;
  k.fblock_first_tile = d.fblock_first_tile;
  k.n_feat_blocks = d.n_feat_blocks;
  k.feat_touched = d.feat_touched;
  k.status = a.status;
  const int resident = resident_grid((const void*)dedup_compact_kernel, kCellThreads, num_sms);
  const int64_t ngroups = (ncells + kGroupCells - 1) / kGroupCells;
  const int64_t rounds =  // of all entries, if they were in one group
      (a.H * (a.cap_prev + a.ecap) + kCompactRound - 1) / kCompactRound;
  int64_t slices = (kCompactOversplit * (int64_t)resident + ngroups - 1) / ngroups;
  if (slices > rounds) slices = rounds;
  k.slices = (int32_t)(slices > kCompactMaxSlices ? kCompactMaxSlices : slices);
  const int64_t fix = (a.ecap + kIlp * kCellThreads - 1) / (kIlp * kCellThreads);
  const int64_t fix_ctas = resident / a.H > 1 ? resident / a.H : 1;
  k.fix_ctas = (int32_t)(fix < fix_ctas ? fix : fix_ctas);
  const int64_t items = ngroups * k.slices, fixes = (int64_t)a.H * k.fix_ctas;
  const int grid = fitted_grid((const void*)dedup_compact_kernel, kCellThreads, num_sms,
                               items > fixes ? items : fixes);
  dedup_compact_kernel<<<grid, kCellThreads, 0, st>>>(k);
  return cudaGetLastError();
}

}  // namespace agnes
