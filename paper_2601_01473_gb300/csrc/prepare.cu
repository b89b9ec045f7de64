// prepare.cu -- agnes_prepare_hyperbatch: one hyperbatch (Algorithm 1,
// Sec. 3.5) on the caller's stream:
//   bucket the targets by (tile, minibatch)                   [sample.cu]
//   for each hop: scan min(deg, k) of the dst lists to indptr, sample in
//                 bucket order                                [sample.cu]
//                 bucket the samples, dedup + relabel, carry the bucket
//                                                             [dedup.cu]
//   gather the final bucket's rows block by block             [gather_hbm.cu]
// Everything is sized for the worst case up front (per-minibatch capacities
// cap_h = min(N, B * prod(1 + k))), so no kernel's launch waits on a count
// from the device and the host synchronises only when a view is fetched.
// With the graph resident the sequence is captured once per hyperbatch shape
// and replayed as one CUDA graph launch.
#include <string.h>

#include <utility>
#include <vector>

#include "ctx.h"

using namespace agnes;

namespace agnes {
namespace {
// A hyperbatch's start, one launch: the targets into the node lists (unless
// targets is null: they were copied from host memory), the sampling key, and
// the readback block cleared but for the targets' frontier sizes.  What a node
// of the sequence costs a small hyperbatch is its place in the chain (about 3 us
// each): with this, one copy of the readback block instead of five, counters
// that their scan clears and block statistics taken from the bucket's offsets,
// 1 x 1024 targets at [15, 10, 5] went from 289 to 272 us and 16 x 1024 from 671
// to 653.
struct BeginArgs {
  const int32_t* targets;  // H x B
  int32_t* nodes;          // H x capK
  int64_t capK;
  int32_t H, B;
  uint64_t* key;
  uint64_t seed, first_gid;
  int32_t* back;
  int64_t back_words;
};

__global__ void __launch_bounds__(256) begin_kernel(BeginArgs a) {
  grid_dep_wait();
  const int64_t i0 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  if (i0 == 0) {
    a.key[0] = a.seed;
    a.key[1] = a.first_gid;
  }
  // word 0 is the status; words 1 .. H are |dst_0| of every minibatch
  for (int64_t i = i0; i < a.back_words; i += stride) a.back[i] = i >= 1 && i <= a.H ? a.B : 0;
  if (!a.targets) return;
  const int64_t n = (int64_t)a.H * a.B;
  for (int64_t i = i0; i < n; i += stride) {
    const int64_t j = i / a.B;
    a.nodes[j * a.capK + (i - j * a.B)] = a.targets[i];
  }
}
}  // namespace
}  // namespace agnes

void free_workspace(Workspace* w) {
  cudaFree(w->nodes);
  for (int b = 0; b < 2; ++b) {
    cudaFree(w->fb_id[b]);
    cudaFree(w->fb_pos[b]);
    cudaFree(w->fcell_off[b]);
  }
  cudaFree(w->fcnt);
  cudaFree(w->scnt);
  cudaFree(w->soff);
  cudaFree(w->nfcnt);
  cudaFree(w->newcnt);
  cudaFree(w->newbase);
  cudaFree(w->back);
  cudaFree(w->noutbase);
  for (int h = 0; h < AGNES_MAX_HOPS; ++h) {
    cudaFree(w->indptr[h]);
    cudaFree(w->col[h]);
  }
  cudaFree(w->nbr);
  cudaFree(w->scell);
  cudaFree(w->srank);
  cudaFree(w->sb);
  cudaFree(w->tmp);
  cudaFree(w->hset);
  cudaFree(w->q_ctl);
  cudaFree(w->q_dense);
  cudaFree(w->tmp_id);
  cudaFree(w->tmp_pos);
  cudaFree(w->indptr_scratch);
  cudaFree(w->flat_scratch);
  cudaFree(w->feats_out);
  cudaFree(w->scan_scratch);
  cudaFree(w->cols_scratch);
  cudaFree(w->distinct);
  cudaFree(w->key);
  if (w->h_back) cudaFreeHost(w->h_back);
  *w = Workspace();
}

template <typename T>
static cudaError_t dalloc(T** p, int64_t n) {
  return cudaMalloc((void**)p, sizeof(T) * (size_t)(n > 0 ? n : 1));
}

static agnes_status ensure_workspace(agnes_ctx* ctx, int32_t H, int32_t B, const int32_t* fan,
                                     int32_t K, const int64_t* cap) {
  Workspace& w = ctx->ws;
  bool same = w.valid && w.H == H && w.B == B && w.K == K;
  for (int h = 0; same && h < K; ++h) same = w.fan[h] == fan[h];
  if (same) return AGNES_OK;
  cudaDeviceSynchronize();
  free_workspace(&w);
  ctx->ws_gen += 1;  // launch sequences captured over the old buffers are stale
  w.H = H;
  w.B = B;
  w.K = K;
  for (int h = 0; h < K; ++h) w.fan[h] = fan[h];
  for (int h = 0; h <= K; ++h) w.cap[h] = cap[h];
  w.capK = cap[K];
  w.ecap_max = 0;
  w.cap_prev_max = 0;
  for (int h = 0; h < K; ++h) {
    const int64_t e = cap[h] * fan[h];
    if (e > w.ecap_max) w.ecap_max = e;
    if (cap[h] > w.cap_prev_max) w.cap_prev_max = cap[h];
  }
  const int64_t T = ctx->bt.T;
  const int64_t cells = T * H;
  const int64_t rows = (int64_t)H * w.capK;
  const int64_t edges = (int64_t)H * w.ecap_max;
  const int64_t scan_elems = scan_scratch_elems(T);

#define WA(p, n)                                                                             \
  do {                                                                                       \
    if (dalloc(&(p), (n)) != cudaSuccess) {                                                  \
      cudaGetLastError();                                                                    \
      free_workspace(&w);                                                                    \
      set_err(ctx, "out of device memory allocating %s (%lld elements)", #p, (long long)(n)); \
      return AGNES_ENOMEM;                                                                   \
    }                                                                                        \
  } while (0)

  WA(w.nodes, rows);
  for (int b = 0; b < 2; ++b) {
    WA(w.fb_id[b], rows);
    WA(w.fb_pos[b], rows);
    WA(w.fcell_off[b], cells + 1);
  }
  WA(w.fcnt, cells);
  WA(w.scnt, cells);
  WA(w.soff, cells + 1);
  WA(w.nfcnt, cells);
  WA(w.newcnt, cells);
  WA(w.newbase, cells);
  w.back_bytes = back_stats_offset(K, H) + sizeof(int64_t) * (size_t)(K + 1);
  {
    uint8_t* p = nullptr;
    WA(p, (int64_t)w.back_bytes);
    w.back = p;
    const Back b = back_at(p, K, H);
    w.status = b.status;
    w.nsz = b.nsz;
    w.ecnt = b.ecnt;
    w.srcsz = b.srcsz;
    w.stats = b.stats;
  }
  WA(w.noutbase, cells);
  for (int h = 0; h < K; ++h) {
    WA(w.indptr[h], (int64_t)H * (cap[h] + 1));
    WA(w.col[h], (int64_t)H * cap[h] * fan[h]);
  }
  WA(w.nbr, edges);
  WA(w.scell, edges);
  WA(w.srank, edges);
  WA(w.sb, edges);
  WA(w.tmp, rows + edges);
  WA(w.q_ctl, 2);
  WA(w.q_dense, (rows + edges) / (kDedupLaneMax + 1) + 1);
  w.hset_elems = 0;
  for (int h = 0; h < K; ++h) {
    int32_t l2 = 0, g = 0;
    const int64_t e = huge_fanout_tables(fan[h], ctx->num_sms, &l2, &g);
    if (e > w.hset_elems) w.hset_elems = e;
  }
  if (w.hset_elems > 0) WA(w.hset, w.hset_elems);
  WA(w.tmp_id, (int64_t)H * B);
  WA(w.tmp_pos, (int64_t)H * B);
  const int64_t indptr_elems = indptr_scratch_elems(H, w.cap_prev_max);
  WA(w.indptr_scratch, indptr_elems);
  w.flat_elems = flat_scan_scratch_elems(cells);
  WA(w.flat_scratch, w.flat_elems);
  {
    uint8_t* f = nullptr;
    WA(f, rows * ctx->row_bytes);
    w.feats_out = f;
  }
  WA(w.scan_scratch, scan_elems);
  WA(w.cols_scratch, cell_scans_scratch_elems(T, H));
  WA(w.distinct, 1);
  WA(w.key, 2);
#undef WA
  if (cudaMallocHost(&w.h_back, w.back_bytes) != cudaSuccess) {
    cudaGetLastError();
    w.h_back = nullptr;
    free_workspace(&w);
    set_err(ctx, "out of pinned host memory");
    return AGNES_ENOMEM;
  }
  if (cudaMemset(w.scan_scratch, 0, sizeof(int64_t) * scan_elems) != cudaSuccess ||
      cudaMemset(w.indptr_scratch, 0, sizeof(uint64_t) * indptr_elems) != cudaSuccess ||
      cudaMemset(w.fcnt, 0, sizeof(int32_t) * cells) != cudaSuccess ||
      cudaMemset(w.scnt, 0, sizeof(int32_t) * cells) != cudaSuccess ||
      cudaMemset(w.flat_scratch, 0, sizeof(uint64_t) * w.flat_elems) != cudaSuccess ||
      // the hyperbatch may run on a stream that does not wait for this one
      cudaStreamSynchronize(cudaStreamLegacy) != cudaSuccess) {
    free_workspace(&w);
    set_err(ctx, "cudaMemset failed");
    return AGNES_ECUDA;
  }
  w.valid = true;
  return AGNES_OK;
}

void swap_hyperbatch_state(agnes_ctx* ctx, agnes_ctx::Spare& o) {
  std::swap(ctx->ws, o.ws);
  std::swap(ctx->lg, o.lg);
  std::swap(ctx->ws_gen, o.ws_gen);
  std::swap(ctx->done, o.done);
  std::swap(ctx->pipe_st, o.pipe_st);
  std::swap(ctx->cur, o.cur);
  std::swap(ctx->prepared, o.prepared);
  std::swap(ctx->synced, o.synced);
}

void rotate_hyperbatch_state(agnes_ctx* ctx) {
  swap_hyperbatch_state(ctx, ctx->spares[0]);
  for (int i = 0; i + 2 < ctx->pipe_depth; ++i) std::swap(ctx->spares[i], ctx->spares[i + 1]);
}

static agnes_status make_one_spare(agnes_ctx* ctx, agnes_ctx::Spare& o) {
  if (o.done) return AGNES_OK;
  const unsigned f = cudaEventDisableTiming;
  if (cudaEventCreateWithFlags(&o.done, f) != cudaSuccess ||
      cudaStreamCreateWithFlags(&o.pipe_st, cudaStreamNonBlocking) != cudaSuccess) {
    cudaGetLastError();
    set_err(ctx, "creating a further hyperbatch's events or streams failed");
    return AGNES_ECUDA;
  }
  o.lg.mode = ctx->lg.mode;
  return AGNES_OK;
}

agnes_status make_spare_state(agnes_ctx* ctx, int32_t depth) {
  for (int i = 0; i + 1 < depth; ++i) {
    const agnes_status rc = make_one_spare(ctx, ctx->spares[i]);
    if (rc != AGNES_OK) return rc;
  }
  const unsigned f = cudaEventDisableTiming;
  if ((!ctx->pipe_st && cudaStreamCreateWithFlags(&ctx->pipe_st, cudaStreamNonBlocking) !=
                            cudaSuccess) ||
      (!ctx->pipe_in && cudaEventCreateWithFlags(&ctx->pipe_in, f) != cudaSuccess)) {
    cudaGetLastError();
    set_err(ctx, "creating the pipeline's stream or event failed");
    return AGNES_ECUDA;
  }
  return AGNES_OK;
}

void free_spare_state(agnes_ctx* ctx) {
  for (agnes_ctx::Spare& o : ctx->spares) {
    drop_launch_graph(&o.lg);
    if (o.lg.cap) cudaStreamDestroy(o.lg.cap);
    o.lg.cap = nullptr;
    free_workspace(&o.ws);
    if (o.done) cudaEventDestroy(o.done);
    if (o.pipe_st) cudaStreamDestroy(o.pipe_st);
    const int32_t mode = o.lg.mode;
    o = agnes_ctx::Spare();
    o.lg.mode = mode;
  }
}

void drop_launch_graph(agnes_ctx::LaunchGraph* g) {
  if (g->exec) cudaGraphExecDestroy(g->exec);
  if (g->graph) cudaGraphDestroy(g->graph);
  g->exec = nullptr;
  g->graph = nullptr;
  g->n_marks = 0;
}

// Enqueues one hyperbatch on st behind its begin_kernel: the bucketing of the targets, K hops of sampling
// and dedup, the feature gather, the statistics and the size read-back.
// mark_flags is cudaEventRecordExternal while the sequence is being captured,
// so the phase events become event-record nodes of the graph; *n_marks gets
// the number of phase events recorded.
static agnes_status enqueue_hyperbatch(agnes_ctx* ctx, const int32_t* fanouts, int32_t K,
                                       const int64_t* cap, int ring, unsigned mark_flags,
                                       cudaStream_t st, int* n_marks) {
  agnes_status rc = AGNES_OK;
  Workspace& w = ctx->ws;
  const int32_t H = w.H, B = w.B;
  const int32_t T = (int32_t)ctx->bt.T;
  const int64_t cells = (int64_t)T * H;
  const int nsm = ctx->num_sms;
  int ph = 0;
  // a phase boundary; with AGNES_PROFILE_GATHER only the gather's two count
  auto mark = [&](bool gather_edge = false) {
    if (ctx->profiling == AGNES_PROFILE_PHASES ||
        (ctx->profiling == AGNES_PROFILE_GATHER && gather_edge))
      cudaEventRecordWithFlags(ctx->ev[ring][ph++], st, mark_flags);
  };

  mark();
  CK(ctx, launch_bucket_targets(w.nodes, w.capK, H, B, (int32_t)ctx->N, ctx->bt.tile_first,
                                ctx->bt.chunk_tile, T, w.fcnt, w.fcell_off[0], w.tmp_id, w.tmp_pos,
                                w.fb_id[0], w.fb_pos[0], w.flat_scratch, w.status, nsm, st));
  int cur = 0;
  for (int h = 0; h < K; ++h) {
    mark();
    HopArgs a;
    a.offsets = ctx->offsets;
    a.offsets_bits = ctx->offsets_bits;
    a.indices = ctx->indices;
    a.N = (int32_t)ctx->N;
    a.tile_first = ctx->bt.tile_first;
    a.chunk_tile = ctx->bt.chunk_tile;
    a.T = T;
    a.H = H;
    a.capK = w.capK;
    a.cap_prev = cap[h];
    a.ecap = cap[h] * fanouts[h];
    a.k = fanouts[h];
    a.hop = h + 1;
    a.key = w.key;
    a.status = w.status;
    a.hset = w.hset;
    huge_fanout_tables(fanouts[h], nsm, &a.hset_log2, &a.hset_grid);
    const bool frontier_sampled = ctx->frontier_mode == AGNES_FRONTIER_SAMPLED && h + 1 < K;
    a.sb_packed = a.ecap <= kPackedEdgeMax;
    int32_t* nsz_prev = w.nsz + (int64_t)h * H;
    int32_t* ecnt = w.ecnt + (int64_t)h * H;
    CK(ctx, launch_sample_indptr(a, w.nodes, nsz_prev, w.indptr[h], ecnt, w.indptr_scratch, nsm,
                                 st));
    mark();
    if (ctx->topo.on) {
      rc = fill_streamed(ctx, a, cur, h, st);
      if (rc != AGNES_OK) return rc;
    } else {
      FillRange r;
      r.cell_lo = 0;
      r.cell_hi = cells;
      const agnes_ctx::Topo& tp = ctx->topo;
      if (tp.cache) {  // requests per block run, then cached blocks from HBM, others in place
        CK(ctx, launch_count_cache_requests(w.fcell_off[cur], T, H, ctx->bt.tile_adj_start,
                                            ctx->bt.tile_adj_block, tp.d_slot, tp.d_acc,
                                            tp.d_cached, w.status, st));
        r.tile_adj_block = ctx->bt.tile_adj_block;
        r.blk_slot = tp.d_slot;
        r.blk_e0 = ctx->bt.blk_e0;
        r.gbuf = tp.gbuf;
        r.epb = tp.epb;
        r.bb = ctx->adj_block_bytes;
        r.in_place_fallback = true;
      }
      CK(ctx, launch_sample_fill(a, w.fb_id[cur], w.fb_pos[cur], w.fcell_off[cur], w.indptr[h],
                                 w.nbr, w.scnt, w.scell, w.srank, r, nsm, st));
    }
    mark();
    DedupBufs d;
    d.nbr = w.nbr;
    d.ecnt = ecnt;
    d.scell = w.scell;
    d.srank = w.srank;
    d.scnt = w.scnt;
    d.soff = w.soff;
    d.sb = w.sb;
    d.tmp = w.tmp;
    d.q_dense = w.q_dense;
    d.q_ctl = w.q_ctl;
    d.indptr_scratch = w.indptr_scratch;
    d.run_first_tile = ctx->bt.run_first_tile;
    d.n_runs = ctx->bt.n_starts;
    d.touched = w.stats + h;
    d.fb_id = w.fb_id[cur];
    d.fb_pos = w.fb_pos[cur];
    d.fcell_off = w.fcell_off[cur];
    d.newcnt = w.newcnt;
    d.newbase = w.newbase;
    d.nfcnt = w.nfcnt;
    d.nfcell_off = w.fcell_off[1 - cur];
    d.nfb_id = w.fb_id[1 - cur];
    d.nfb_pos = w.fb_pos[1 - cur];
    d.nsz_prev = nsz_prev;
    d.nsz_next = w.nsz + (int64_t)(h + 1) * H;
    d.srcsz = w.srcsz + (int64_t)h * H;
    d.noutbase = w.noutbase;
    d.frontier_sampled = frontier_sampled;
    d.nodes = w.nodes;
    d.col = w.col[h];
    d.cols_scratch = w.cols_scratch;
    d.flat_scratch = w.flat_scratch;
    if (h + 1 == K) {
      d.fblock_first_tile = ctx->bt.fblock_first_tile;
      d.n_feat_blocks = ctx->bt.n_feat_blocks;
      d.feat_touched = w.stats + K;
    }
    CK(ctx, launch_dedup(a, d, nsm, st));
    cur = 1 - cur;
  }
  mark(true);
  if (ctx->features_on_host) {
    rc = gather_streamed(ctx, cur, st);
    if (rc != AGNES_OK) return rc;
  } else {
    CK(ctx, launch_gather(ctx->features, ctx->N * ctx->row_bytes, ctx->row_bytes, w.fb_id[cur],
                          w.fb_pos[cur], w.fcell_off[cur] + cells, H * w.capK, w.feats_out,
                          w.status, nsm, st));
  }
  mark(true);
  CK(ctx, cudaMemcpyAsync(w.h_back, w.back, w.back_bytes, cudaMemcpyDeviceToHost, st));
  if (ctx->topo.cache)
    CK(ctx, cudaMemcpyAsync(ctx->topo.h_cached, ctx->topo.d_cached, sizeof(unsigned long long),
                            cudaMemcpyDeviceToHost, st));
  *n_marks = ph;
  return AGNES_OK;
}

// Whether a kernel on `device` can read int32 values at p: its own device memory
// or managed memory, aligned to them (a copy takes any address).
static bool device_can_read(const void* p, int device) {
  if ((uintptr_t)p % sizeof(int32_t) != 0) return false;
  cudaPointerAttributes attr;
  if (cudaPointerGetAttributes(&attr, p) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return attr.type == cudaMemoryTypeManaged ||
         (attr.type == cudaMemoryTypeDevice && attr.device == device);
}

// Whether work enqueued on st is being captured (by the caller's own graph
// capture); an unknown state counts as captured, so the sequence is enqueued
// as it is.
static bool stream_capturing(cudaStream_t st) {
  cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(st, &cs) != cudaSuccess) {
    cudaGetLastError();
    return true;
  }
  return cs != cudaStreamCaptureStatusNone;
}

// Turns every kernel-to-kernel link of the captured chain (an edge whose
// source has no other successor and whose destination no other predecessor)
// into a programmatic one from the programmatic port: the kernels trigger nothing
// early, so the next kernel is launched as soon as every block of its
// predecessor has exited, and its blocks wait at their first statement
// (grid_dep_wait) for the predecessor's writes to become visible; the launch
// overlaps the predecessor's completion instead of following it.  (Launching
// once all predecessor blocks had merely started was measured slower: the
// waiting blocks took SM slots from the running kernel's tail.)  Edges
// touching other nodes (memsets, copies, event records) keep full
// serialisation.
static cudaError_t make_programmatic(cudaGraph_t graph, int64_t* converted) {
  size_t n = 0;
  cudaError_t e = cudaGraphGetEdges(graph, nullptr, nullptr, nullptr, &n);
  if (e != cudaSuccess || n == 0) return e;
  std::vector<cudaGraphNode_t> from(n), to(n);
  std::vector<cudaGraphEdgeData> data(n);
  e = cudaGraphGetEdges(graph, from.data(), to.data(), data.data(), &n);
  if (e != cudaSuccess) return e;
  std::vector<std::pair<cudaGraphNode_t, int>> outs, ins;  // edge counts per node
  auto bump = [](std::vector<std::pair<cudaGraphNode_t, int>>& v, cudaGraphNode_t nd) {
    for (auto& p : v)
      if (p.first == nd) return ++p.second;
    v.emplace_back(nd, 1);
    return 1;
  };
  auto count = [](const std::vector<std::pair<cudaGraphNode_t, int>>& v, cudaGraphNode_t nd) {
    for (const auto& p : v)
      if (p.first == nd) return p.second;
    return 0;
  };
  for (size_t i = 0; i < n; ++i) {
    bump(outs, from[i]);
    bump(ins, to[i]);
  }
  for (size_t i = 0; i < n; ++i) {
    if (count(outs, from[i]) != 1 || count(ins, to[i]) != 1) continue;
    cudaGraphNodeType tf, tt;
    if ((e = cudaGraphNodeGetType(from[i], &tf)) != cudaSuccess) return e;
    if ((e = cudaGraphNodeGetType(to[i], &tt)) != cudaSuccess) return e;
    if (tf != cudaGraphNodeTypeKernel || tt != cudaGraphNodeTypeKernel) continue;
    if (data[i].type != cudaGraphDependencyTypeDefault || data[i].from_port != 0) continue;
    if ((e = cudaGraphRemoveDependencies(graph, &from[i], &to[i], &data[i], 1)) != cudaSuccess)
      return e;
    cudaGraphEdgeData p;
    memset(&p, 0, sizeof(p));
    p.from_port = cudaGraphKernelNodePortProgrammatic;
    p.type = cudaGraphDependencyTypeProgrammatic;
    if ((e = cudaGraphAddDependencies(graph, &from[i], &to[i], &p, 1)) != cudaSuccess) return e;
    *converted += 1;
  }
  return cudaSuccess;
}

// The resident path as one graph launch.  The launch sequence is captured on
// a private stream the first time a hyperbatch shape (H, B, fanouts, frontier
// mode, profiling, workspace) is seen, and replayed for every later hyperbatch
// of that shape: everything that varies between them (the targets, the seed,
// the minibatch ids) is in device memory by then.  With profiling on, the
// captured phase-event nodes are pointed at this prepare's ring slot.
static agnes_status launch_graphed(agnes_ctx* ctx, const int32_t* fanouts, int32_t K,
                                   const int64_t* cap, int ring, cudaStream_t st,
                                   int* n_marks) {
  agnes_ctx::LaunchGraph& g = ctx->lg;
  const Workspace& w = ctx->ws;
  bool same = g.exec && g.H == w.H && g.B == w.B && g.K == K &&
              g.frontier_mode == ctx->frontier_mode && g.profiling == ctx->profiling &&
              g.ws_gen == ctx->ws_gen && g.built_mode == g.mode;
  for (int h = 0; same && h < K; ++h) same = g.fan[h] == fanouts[h];
  if (!same) {
    drop_launch_graph(&g);
    if (!g.cap) CK(ctx, cudaStreamCreateWithFlags(&g.cap, cudaStreamNonBlocking));
    CK(ctx, cudaStreamBeginCapture(g.cap, cudaStreamCaptureModeRelaxed));
    int nm = 0;
    const agnes_status rc =
        enqueue_hyperbatch(ctx, fanouts, K, cap, ring, cudaEventRecordExternal, g.cap, &nm);
    cudaGraph_t graph = nullptr;
    const cudaError_t e = cudaStreamEndCapture(g.cap, &graph);
    if (rc != AGNES_OK || e != cudaSuccess) {
      if (graph) cudaGraphDestroy(graph);
      cudaGetLastError();
      if (rc != AGNES_OK) return rc;
      set_err(ctx, "capturing the launch sequence failed: %s", cudaGetErrorString(e));
      return AGNES_ECUDA;
    }
    g.graph = graph;
    g.programmatic_edges = 0;
    if (g.mode == AGNES_LAUNCH_GRAPH_PDL) CK(ctx, make_programmatic(graph, &g.programmatic_edges));
    CK(ctx, cudaGraphInstantiate(&g.exec, graph, 0));
    if (ctx->profiling) {
      size_t n = 0;
      CK(ctx, cudaGraphGetNodes(graph, nullptr, &n));
      std::vector<cudaGraphNode_t> nodes(n);
      CK(ctx, cudaGraphGetNodes(graph, nodes.data(), &n));
      for (int i = 0; i < nm; ++i) g.phase_node[i] = nullptr;
      for (cudaGraphNode_t nd : nodes) {
        cudaGraphNodeType t;
        CK(ctx, cudaGraphNodeGetType(nd, &t));
        if (t != cudaGraphNodeTypeEventRecord) continue;
        cudaEvent_t ev = nullptr;
        CK(ctx, cudaGraphEventRecordNodeGetEvent(nd, &ev));
        for (int i = 0; i < nm; ++i)
          if (ctx->ev[ring][i] == ev) g.phase_node[i] = nd;
      }
      for (int i = 0; i < nm; ++i) {
        if (!g.phase_node[i]) {
          drop_launch_graph(&g);
          set_err(ctx, "phase event %d is missing from the captured launch sequence", i);
          return AGNES_ECUDA;
        }
      }
    }
    g.n_marks = nm;
    g.H = w.H;
    g.B = w.B;
    g.K = K;
    for (int h = 0; h < K; ++h) g.fan[h] = fanouts[h];
    g.frontier_mode = ctx->frontier_mode;
    g.built_mode = g.mode;
    g.profiling = ctx->profiling;
    g.ws_gen = ctx->ws_gen;
    g.captures += 1;
  }
  if (g.profiling)
    for (int i = 0; i < g.n_marks; ++i)
      CK(ctx, cudaGraphExecEventRecordNodeSetEvent(g.exec, g.phase_node[i], ctx->ev[ring][i]));
  CK(ctx, cudaGraphLaunch(g.exec, st));
  g.launches += 1;
  *n_marks = g.n_marks;
  return AGNES_OK;
}

extern "C" {

agnes_status agnes_prepare_hyperbatch(agnes_ctx* ctx, const int32_t* targets, int32_t H,
                                      int32_t B, const int32_t* fanouts, int32_t K,
                                      uint64_t seed, uint64_t first_minibatch_id,
                                      void* cuda_stream) {
  if (!ctx) {
    set_err(nullptr, "ctx is NULL");
    return AGNES_EINVAL;
  }
  if (!targets || !fanouts) {
    set_err(ctx, "targets and fanouts must be non-NULL");
    return AGNES_EINVAL;
  }
  if (H < 1 || H > 65535 || B < 1 || K < 1 || K > AGNES_MAX_HOPS) {
    set_err(ctx, "need 1 <= H <= 65535, B >= 1, 1 <= K <= %d", AGNES_MAX_HOPS);
    return AGNES_EINVAL;
  }
  if (B > ctx->N) {
    set_err(ctx, "B = %d distinct targets exceed N = %lld", B, (long long)ctx->N);
    return AGNES_EINVAL;
  }
  int64_t cap[AGNES_MAX_HOPS + 1];
  cap[0] = B;
  for (int h = 0; h < K; ++h) {
    if (fanouts[h] < 1 || fanouts[h] > AGNES_MAX_FANOUT) {
      set_err(ctx, "fanouts[%d] = %d outside [1, %d]", h, fanouts[h], AGNES_MAX_FANOUT);
      return AGNES_EINVAL;
    }
    const int64_t grown = cap[h] * (1 + (int64_t)fanouts[h]);
    cap[h + 1] = grown < ctx->N ? grown : ctx->N;
  }
  const int64_t lim = ((int64_t)1 << 31) - 1;
  for (int h = 0; h < K; ++h) {
    if ((int64_t)H * cap[h] * fanouts[h] > lim) {
      set_err(ctx, "H x edge capacity of hop %d exceeds 2^31", h + 1);
      return AGNES_ERANGE;
    }
  }
  if ((int64_t)H * cap[K] > lim) {
    set_err(ctx, "H x node capacity (%lld) exceeds 2^31", (long long)(H * cap[K]));
    return AGNES_ERANGE;
  }
  if ((int64_t)H * ctx->bt.T >= lim) {  // cell indices are 31-bit in the kernels
    set_err(ctx, "H x tiles (%lld) exceeds 2^31", (long long)(H * ctx->bt.T));
    return AGNES_ERANGE;
  }
  DeviceGuard dg(ctx->device);
  if (!dg.ok()) {
    set_err(ctx, "cudaSetDevice(%d) failed", ctx->device);
    return AGNES_ECUDA;
  }
  const cudaStream_t caller = (cudaStream_t)cuda_stream;
  const bool capturing = stream_capturing(caller);
  const bool resident = !ctx->features_on_host && !ctx->topo.on;
  const bool pipelined = ctx->pipe_depth > 1 && resident && !capturing;
  // the least recently used set of per-hyperbatch state
  if (pipelined) rotate_hyperbatch_state(ctx);
  const cudaStream_t st = pipelined ? ctx->pipe_st : caller;
  ctx->prepared = false;  // also if the workspace cannot be allocated: the last one is gone
  ctx->synced = false;
  agnes_status rc = ensure_workspace(ctx, H, B, fanouts, K, cap);
  if (rc != AGNES_OK) return rc;
  Workspace& w = ctx->ws;
  if (ctx->profiling && !ctx->ev_created) {
    for (int r = 0; r < kEventRing; ++r)
      for (int i = 0; i <= kMaxPhases; ++i) CK(ctx, cudaEventCreate(&ctx->ev[r][i]));
    ctx->ev_created = true;
  }
  const int ring = (int)(ctx->n_prepared % kEventRing);
  ctx->n_phases[ring] = 0;
  // a prepare on another stream than the last one on these buffers still runs
  // after it (a caller's own capture orders its replays itself)
  if (ctx->n_prepared > 0 && !capturing) CK(ctx, cudaStreamWaitEvent(caller, ctx->done, 0));
  if (!capturing) {
    rc = update_topology_cache(ctx, caller);
    if (rc != AGNES_OK) return rc;
  }
  // the targets are read on the caller's stream, whatever the hyperbatch runs on:
  // what the stream does next may overwrite or free them
  BeginArgs b;
  b.targets = device_can_read(targets, ctx->device) ? targets : nullptr;
  if (!b.targets)
    CK(ctx, cudaMemcpy2DAsync(w.nodes, sizeof(int32_t) * w.capK, targets, sizeof(int32_t) * B,
                              sizeof(int32_t) * B, H, cudaMemcpyDefault, caller));
  b.nodes = w.nodes;
  b.capK = w.capK;
  b.H = H;
  b.B = B;
  b.key = w.key;
  b.seed = seed;
  b.first_gid = first_minibatch_id;
  b.back = (int32_t*)w.back;
  b.back_words = (int64_t)(w.back_bytes / sizeof(int32_t));
  const int64_t most = b.back_words > (int64_t)H * B ? b.back_words : (int64_t)H * B;
  begin_kernel<<<fitted_grid((const void*)begin_kernel, 256, ctx->num_sms, (most + 255) / 256), 256,
                 0, caller>>>(b);
  CK(ctx, cudaGetLastError());
  if (pipelined) {
    CK(ctx, cudaEventRecord(ctx->pipe_in, caller));
    CK(ctx, cudaStreamWaitEvent(st, ctx->pipe_in, 0));
  }
  int n_marks = 0;
  if (resident && ctx->lg.mode != AGNES_LAUNCH_DIRECT && !capturing)
    rc = launch_graphed(ctx, fanouts, K, cap, ring, st, &n_marks);
  else
    rc = enqueue_hyperbatch(ctx, fanouts, K, cap, ring, cudaEventRecordDefault, st, &n_marks);
  if (rc != AGNES_OK) {
    w.valid = false;  // a sequence cut short may have left counters set: start from a new one
    return rc;
  }
  // inside a caller's capture nothing has run yet: the caller orders its
  // replays, and there are no phase times to read
  if (!capturing) CK(ctx, cudaEventRecord(ctx->done, st));
  ctx->n_phases[ring] = ctx->profiling && !capturing ? n_marks - 1 : 0;
  ctx->n_prepared += 1;
  ctx->cur = K & 1;  // the frontier buffers swap once per hop
  ctx->prepared = true;
  return AGNES_OK;
}

}  // extern "C"
