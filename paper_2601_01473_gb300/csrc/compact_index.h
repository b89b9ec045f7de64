// compact_index.h -- index arithmetic of the compaction of the next frontier
// bucket (dedup.cu), apart from the kernel so that it can be checked at sizes
// that no test would allocate.
//
// A hyperbatch may have up to 2^31 - 1 frontier entries and as many sampled
// ones, so a place in tmp (frontier and sampled entries before it) and the
// first entry of a CTA's next round can pass 2^31: the one is kept in 64 bits,
// where its complement can mark it as one in tmp (a 32-bit place and a flag of its
// own cost 1 x 1024 targets on 10M nodes 219 -> 224 us), the other is unsigned.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace agnes {

constexpr int kCellThreads = 128;  // threads per CTA of the compaction
constexpr int kCompactIlp = 2;  // bucket entries per thread and round (4 and 8 measured slower)
constexpr int kCompactMaxSlices = 256;  // of a group, binding where a graph has a few tiles:
                                        // hop 2 of 32 x 1024 targets on 20k nodes with 64,
                                        // 256, 1024: dedup 351, 344, 344 us
constexpr int kCompactRound = kCompactIlp * kCellThreads;

// Where a cell's next-frontier entries start in tmp: behind its `fo` frontier
// and `so` sampled predecessors.
__host__ __device__ inline int64_t tmp_base(int32_t fo, int32_t so) {
  return (int64_t)fo + so;
}

// A thread's first entry of a group that starts at k0, and of its next round.
__host__ __device__ inline uint32_t compact_first(int32_t k0, int32_t slice, int32_t thread) {
  return (uint32_t)k0 + (uint32_t)(slice * kCompactRound + thread);
}
__host__ __device__ inline uint32_t compact_next(uint32_t k, int32_t slices) {
  return k + (uint32_t)(slices * kCompactRound);
}

}  // namespace agnes
