// gather_hbm.cu -- block-wise feature gathering from HBM-resident features
// (Algorithm 1's gathering loop, Sec. 3.4 (2)).
//
// The final frontier bucket lists every gathered node once per minibatch, in
// (tile, minibatch, id) order, with its output row.  Tiles never straddle a
// feature block, so walking the bucket in order visits each feature block
// once for all minibatches: a row requested by several minibatches is read
// from HBM once and served from L2 afterwards.  Rows are copied as 16-byte
// vectors (bit-exact, no float conversion); a group of row_bytes/16 lanes
// moves one row, each lane keeping U rows in flight; output stores are
// streaming (evict-first) so they do not push the feature rows out of L2.
#include "common.cuh"
#include "internal.h"

namespace agnes {

namespace {

constexpr int kThreads = 256;
// CTAs per SM of the gather (0: as many as fit) and rows in flight per lane.
// A few CTAs with several rows each keep HBM busy and leave the rest of each
// SM to the kernels of the next hyperbatch, which run beside the gather when
// two hyperbatches are in flight.
constexpr int kGatherCtasPerSm = 3;
constexpr int kU = 8;
// Vectors from which a row has a warp of its own, and whole numbers of which take
// the kernel for whole rows.
constexpr int kWideRow = 176;
constexpr int kWideWhole = 128;

// LPR lanes per row, row = LPR 16-byte vectors, U rows in flight per lane.
template <int LPR, int U>
__global__ void __launch_bounds__(kThreads)
gather_vec_kernel(const uint4* __restrict__ feats, const int32_t* __restrict__ fb_id,
                  const int32_t* __restrict__ fb_pos, const int32_t* total_ptr,
                  uint4* __restrict__ out, const int32_t* status) {
  grid_dep_wait();
  if (failed(status)) return;
  constexpr int kRowsPerWarp = 32 / LPR;
  constexpr int kStep = kRowsPerWarp * U;
  const int64_t total = *total_ptr;
  const int lane = lane_id();
  const int sub = lane / LPR, l = lane % LPR;
  const int64_t warp0 = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t r0 = warp0 * kStep; r0 < total; r0 += nwarps * kStep) {
    uint4 v[U];
    int32_t g[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int64_t i = r0 + u * kRowsPerWarp + sub;
      g[u] = -1;
      if (i < total) {
        const int32_t id = __ldg(fb_id + i);
        g[u] = __ldg(fb_pos + i);
        v[u] = __ldg(feats + (int64_t)id * LPR + l);
      }
    }
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (g[u] >= 0) __stcs(out + (int64_t)g[u] * LPR + l, v[u]);
  }
}

// Rows of any number of 16-byte vectors.  A warp takes R consecutive bucket
// entries and walks their R * vecs vectors as one range, lane after lane, with
// U loads in flight per lane before their stores, so that neither a short row
// (idle lanes) nor a row of 25 vectors (a nearly empty last round) costs
// bandwidth (13 minibatches of 1000 targets, rows of 25 vectors: 264 -> 239 us a
// hyperbatch against a warp per row; 438k rows alone, of 2 vectors 76 -> 14 us, 5 82 ->
// 20, 12 98 -> 39, 25 119 -> 69, 40 174 -> 100, 64 194 -> 135, 128 262 -> 264).
template <int U>
__global__ void __launch_bounds__(kThreads)
gather_any_kernel(const uint4* __restrict__ feats, uint32_t vecs, int32_t R, uint64_t inv_vecs,
                  const int32_t* __restrict__ fb_id, const int32_t* __restrict__ fb_pos,
                  const int32_t* total_ptr, uint4* __restrict__ out, const int32_t* status) {
  grid_dep_wait();
  if (failed(status)) return;
  const int64_t total = *total_ptr;
  const int lane = lane_id();
  const int64_t warp0 = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t r0 = warp0 * R; r0 < total; r0 += nwarps * R) {
    const int32_t rows = (int32_t)min((int64_t)R, total - r0);
    int32_t id = 0, pos = 0;  // of entry r0 + lane
    if (lane < rows) {
      id = __ldg(fb_id + r0 + lane);
      pos = __ldg(fb_pos + r0 + lane);
    }
    const uint32_t m = (uint32_t)rows * vecs;
    for (uint32_t q0 = 0; q0 < m; q0 += 32 * U) {
      uint4 v[U];
      int64_t to[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const uint32_t q = q0 + 32 * u + lane;
        // q / vecs (see rows_per_range)
        const uint32_t row = R == 1 ? 0u : (uint32_t)((q * inv_vecs) >> 32);
        const int32_t src = __shfl_sync(0xffffffffu, id, row & 31);
        const int32_t dst = __shfl_sync(0xffffffffu, pos, row & 31);
        to[u] = -1;
        if (q < m) {
          const uint32_t c = q - row * vecs;
          v[u] = __ldg(feats + (int64_t)src * vecs + c);
          to[u] = (int64_t)dst * vecs + c;
        }
      }
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (to[u] >= 0) __stcs(out + to[u], v[u]);
    }
  }
}

// Rows of 176 vectors and more have a warp each.  A warp's range of
// gather_any_kernel is one such row, in rounds of 8 loads and 8 stores a lane, and
// takes longer.  438k rows, us (any / whole / odd kernel): 144 vectors 329 / 336 /
// 333, 176: 391 / 416 / 348, 224: 493 / 492 / 411, 255: 590 / 657 / 469, 256: 559 /
// 502 / 536, 257: 642 / 610 / 548, 384: 825 / 745 / 802, 512: 1114 / 997 / 1073, 513:
// 1228 / 1178 / 1069, 625: 1462 / 1608 / 1252, 1024: 2233 / 1995 / 2156.

// A whole number of kWideWhole vectors: the compiler's own unrolling of one
// vector a lane.
__global__ void __launch_bounds__(kThreads)
gather_whole_rows_kernel(const uint4* __restrict__ feats, int64_t vecs,
                         const int32_t* __restrict__ fb_id, const int32_t* __restrict__ fb_pos,
                         const int32_t* total_ptr, uint4* __restrict__ out,
                         const int32_t* status) {
  grid_dep_wait();
  if (failed(status)) return;
  const int64_t total = *total_ptr;
  const int lane = lane_id();
  const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t i = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5; i < total; i += nwarps) {
    const int64_t src = (int64_t)__ldg(fb_id + i) * vecs;
    const int64_t dst = (int64_t)__ldg(fb_pos + i) * vecs;
    for (int64_t c = lane; c < vecs; c += 32) __stcs(out + dst + c, __ldg(feats + src + c));
  }
}

// Any other number: rounds of U loads a lane, the last of them in part.
template <int U>
__global__ void __launch_bounds__(kThreads)
gather_odd_rows_kernel(const uint4* __restrict__ feats, int64_t vecs,
                       const int32_t* __restrict__ fb_id, const int32_t* __restrict__ fb_pos,
                       const int32_t* total_ptr, uint4* __restrict__ out, const int32_t* status) {
  grid_dep_wait();
  if (failed(status)) return;
  const int64_t total = *total_ptr;
  const int lane = lane_id();
  const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t i = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5; i < total; i += nwarps) {
    const uint4* src = feats + (int64_t)__ldg(fb_id + i) * vecs;
    uint4* dst = out + (int64_t)__ldg(fb_pos + i) * vecs;
    for (int64_t c0 = lane; c0 < vecs; c0 += 32 * U) {
      uint4 v[U];
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (c0 + 32 * u < vecs) v[u] = __ldg(src + c0 + 32 * u);
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (c0 + 32 * u < vecs) __stcs(dst + c0 + 32 * u, v[u]);
    }
  }
}

// The 16 bytes at the 16-byte boundary p, of which only those in [lo, hi), the
// feature matrix, are read (the rest are zero).
__device__ __forceinline__ uint4 load_within(uintptr_t p, uintptr_t lo, uintptr_t hi) {
  if (p >= lo && p + 16 <= hi) return __ldg((const uint4*)p);
  uint32_t w[4] = {0, 0, 0, 0};
  for (int i = 0; i < 16; ++i)
    if (p + i >= lo && p + i < hi)
      w[i >> 2] |= (uint32_t)__ldg((const uint8_t*)(p + i)) << (8 * (i & 3));
  return make_uint4(w[0], w[1], w[2], w[3]);
}

// Rows whose size or addresses are not multiples of 16 bytes, but of E (4, 2 or
// 1).  The output row is written as its aligned 16-byte vectors, the first and
// last of them in part; the 16 source bytes of each come from the one or two
// aligned vectors that hold them, shifted by bytes, so a load moves four times
// the bytes of a word copy and more (8 minibatches of 500 targets, rows of 1204
// bytes: 306 -> 277 us a hyperbatch against a copy by words, and 309 by bytes).
// Ranges of R rows as in gather_any_kernel, `vecs` being the most vectors a row
// can touch.
template <int E, int U>
__global__ void __launch_bounds__(kThreads)
gather_shift_kernel(uintptr_t feats, uintptr_t feats_end, int64_t row_bytes, uint32_t vecs,
                    int32_t R, uint64_t inv_vecs, const int32_t* __restrict__ fb_id,
                    const int32_t* __restrict__ fb_pos, const int32_t* total_ptr, uintptr_t out,
                    const int32_t* status) {
  grid_dep_wait();
  if (failed(status)) return;
  const int64_t total = *total_ptr;
  const int lane = lane_id();
  const int64_t warp0 = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5;
  const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t r0 = warp0 * R; r0 < total; r0 += nwarps * R) {
    const int32_t rows = (int32_t)min((int64_t)R, total - r0);
    int32_t id = 0, pos = 0;  // of entry r0 + lane
    if (lane < rows) {
      id = __ldg(fb_id + r0 + lane);
      pos = __ldg(fb_pos + r0 + lane);
    }
    const uint32_t m = (uint32_t)rows * vecs;
    for (uint32_t q0 = 0; q0 < m; q0 += 32 * U) {
      uint4 v0[U], v1[U];
      uintptr_t to[U];   // the output vector
      int32_t from[U];   // its first byte of the row, 0 .. 15
      int32_t until[U];  // one past its last, 0: nothing to write
      int32_t shift[U];  // its first byte's place in v0
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const uint32_t q = q0 + 32 * u + lane;
        const uint32_t row = R == 1 ? 0u : (uint32_t)((q * inv_vecs) >> 32);
        const int32_t src = __shfl_sync(0xffffffffu, id, row & 31);
        const int32_t dst = __shfl_sync(0xffffffffu, pos, row & 31);
        until[u] = 0;
        if (q < m) {
          const uint32_t c = q - row * vecs;
          const uintptr_t s = feats + (uintptr_t)((int64_t)src * row_bytes);
          const uintptr_t d = out + (uintptr_t)((int64_t)dst * row_bytes);
          const int32_t head = (int32_t)(d & 15);
          const int64_t left = row_bytes + head - 16 * (int64_t)c;  // bytes up to the row's end
          if (left > 0) {
            from[u] = c == 0 ? head : 0;
            until[u] = left < 16 ? (int32_t)left : 16;
            to[u] = d - head + 16 * (uintptr_t)c;
            const uintptr_t at = s - head + 16 * (uintptr_t)c;  // byte 0's source
            shift[u] = (int32_t)(at & 15);
            const uintptr_t base = at - shift[u];
            v0[u] = v1[u] = make_uint4(0, 0, 0, 0);
            if (shift[u] + from[u] < 16) v0[u] = load_within(base, feats, feats_end);
            if (shift[u] + until[u] > 16) v1[u] = load_within(base + 16, feats, feats_end);
          }
        }
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        if (until[u] == 0) continue;
        uint32_t w[8] = {v0[u].x, v0[u].y, v0[u].z, v0[u].w, v1[u].x, v1[u].y, v1[u].z, v1[u].w};
        if (shift[u] & 8) {
#pragma unroll
          for (int i = 0; i < 6; ++i) w[i] = w[i + 2];
        }
        if (shift[u] & 4) {
#pragma unroll
          for (int i = 0; i < 5; ++i) w[i] = w[i + 1];
        }
        if constexpr (E < 4) {
#pragma unroll
          for (int i = 0; i < 4; ++i) w[i] = __funnelshift_r(w[i], w[i + 1], 8 * (shift[u] & 3));
        }
        if (from[u] == 0 && until[u] == 16) {
          __stcs((uint4*)to[u], make_uint4(w[0], w[1], w[2], w[3]));
        } else {
#pragma unroll
          for (int i = 0; i < 16; i += E) {
            if (i < from[u] || i >= until[u]) continue;
            const uint32_t x = w[i >> 2] >> (8 * (i & 3));
            if constexpr (E == 4)
              *(uint32_t*)(to[u] + i) = x;
            else if constexpr (E == 2)
              *(uint16_t*)(to[u] + i) = (uint16_t)x;
            else
              *(uint8_t*)(to[u] + i) = (uint8_t)x;
          }
        }
      }
    }
  }
}

// Entries a warp takes at a time: about U vectors per lane, at most 32 (a lane
// holds one entry's id).  With R > 1, vecs <= 16 * U and q < 64 * U, so with
// inv_vecs = ceil(2^32 / vecs) the product q * inv_vecs exceeds q / vecs * 2^32
// by less than q < 2^32 / vecs, and its upper word is q / vecs exactly.
int32_t rows_per_range(int64_t vecs, int U) {
  const int64_t r = (32 * U) / vecs;
  return (int32_t)(r < 1 ? 1 : r > 32 ? 32 : r);
}

uint64_t inverse_of(int64_t vecs) { return ((1ull << 32) + vecs - 1) / vecs; }

// CTAs for at most max_total rows, per_warp of them a warp takes at a time.
int gather_grid(const void* kernel, int ctas_per_sm, int num_sms, int64_t max_total,
                int64_t per_warp) {
  const int64_t per_cta = per_warp * (kThreads / 32);
  const int g = fitted_grid(kernel, kThreads, num_sms, (max_total + per_cta - 1) / per_cta);
  return ctas_per_sm > 0 && g > ctas_per_sm * num_sms ? ctas_per_sm * num_sms : g;
}

template <int E>
cudaError_t launch_gather_shift(const void* feats, int64_t feats_bytes, int64_t row_bytes,
                                const int32_t* fb_id, const int32_t* fb_pos,
                                const int32_t* total, int64_t max_total, void* out,
                                const int32_t* status, int num_sms, cudaStream_t st) {
  constexpr int U = 3;  // 438k rows of 100, 260, 1204, 4100 bytes with 2: 35, 76, 274, 766 us;
                        // with 3: 35, 67, 266, 751; with 4: 39, 78, 331, 934
  const int64_t vecs = (row_bytes + 15 + 15) / 16;  // a row may start anywhere in a vector
  const int32_t R = rows_per_range(vecs, U);
  const auto kernel = gather_shift_kernel<E, U>;
  kernel<<<gather_grid((const void*)kernel, 0, num_sms, max_total, R), kThreads, 0, st>>>(
      (uintptr_t)feats, (uintptr_t)feats + (uintptr_t)feats_bytes, row_bytes, (uint32_t)vecs, R,
      inverse_of(vecs), fb_id, fb_pos, total, (uintptr_t)out, status);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_gather(const void* feats, int64_t feats_bytes, int64_t row_bytes,
                          const int32_t* fb_id, const int32_t* fb_pos, const int32_t* total,
                          int64_t max_total, void* out, const int32_t* status, int num_sms,
                          cudaStream_t st) {
  // what the row size and both addresses are multiples of
  const uint64_t align = (uint64_t)row_bytes | (uintptr_t)feats | (uintptr_t)out;
  if (align % 16 != 0) {
    const auto shift = align % 4 == 0   ? launch_gather_shift<4>
                       : align % 2 == 0 ? launch_gather_shift<2>
                                        : launch_gather_shift<1>;
    return shift(feats, feats_bytes, row_bytes, fb_id, fb_pos, total, max_total, out, status,
                 num_sms, st);
  }
  const int64_t vecs = row_bytes / 16;
  const uint4* f = (const uint4*)feats;
  uint4* o = (uint4*)out;
  const int32_t R = rows_per_range(vecs, kU);
#define AGNES_GRID(KERNEL) \
  gather_grid((const void*)KERNEL, kGatherCtasPerSm, num_sms, max_total, R), kThreads, 0, st
  if (vecs == 8)
    gather_vec_kernel<8, kU><<<AGNES_GRID((gather_vec_kernel<8, kU>))>>>(f, fb_id, fb_pos, total,
                                                                         o, status);
  else if (vecs == 16)
    gather_vec_kernel<16, kU><<<AGNES_GRID((gather_vec_kernel<16, kU>))>>>(f, fb_id, fb_pos, total,
                                                                           o, status);
  else if (vecs == 32)
    gather_vec_kernel<32, kU><<<AGNES_GRID((gather_vec_kernel<32, kU>))>>>(f, fb_id, fb_pos, total,
                                                                           o, status);
  else if (vecs >= kWideRow && vecs % kWideWhole == 0)
    gather_whole_rows_kernel<<<AGNES_GRID(gather_whole_rows_kernel)>>>(f, vecs, fb_id, fb_pos, total,
                                                                       o, status);
  else if (vecs >= kWideRow)
    gather_odd_rows_kernel<4><<<AGNES_GRID(gather_odd_rows_kernel<4>)>>>(f, vecs, fb_id, fb_pos,
                                                                         total, o, status);
  else
    gather_any_kernel<kU><<<AGNES_GRID(gather_any_kernel<kU>)>>>(
        f, (uint32_t)vecs, R, inverse_of(vecs), fb_id, fb_pos, total, o, status);
#undef AGNES_GRID
  return cudaGetLastError();
}

}  // namespace agnes
