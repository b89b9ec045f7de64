"""The compaction's index arithmetic (csrc/compact_index.h) at the largest
hyperbatch that agnes_prepare_hyperbatch accepts, compiled for the host: 2^31 -
1 frontier entries and as many sampled ones."""
import subprocess

from paper_2601_01473_gb300 import build

SOURCE = r"""
#include <cstdio>
#include "compact_index.h"
using namespace agnes;
int main() {
  const int32_t most = 0x7fffffff;
  // the last cell's place in tmp, and the place before it
  printf("%llu\n", (unsigned long long)tmp_base(most, most));
  printf("%llu\n", (unsigned long long)tmp_base(most - 3, most));
  // a group of the last 300 entries in the most slices: every entry once
  const int32_t k0 = most - 300;
  long long seen = 0, sum = 0;
  for (int slice = 0; slice < kCompactMaxSlices; ++slice)
    for (int t = 0; t < kCellThreads; ++t) {
      int rounds = 0;
      for (uint32_t kb = compact_first(k0, slice, t); kb < (uint32_t)most && rounds < 3;
           kb = compact_next(kb, kCompactMaxSlices), ++rounds)
        for (int u = 0; u < kCompactIlp; ++u) {
          const uint32_t k = kb + u * kCellThreads;
          if (k < (uint32_t)most) { ++seen; sum += k - (uint32_t)k0; }
        }
    }
  printf("%lld %lld\n", seen, sum);
}
"""


def test_indexes_at_the_largest_hyperbatch(tmp_path):
    src, exe = tmp_path / "index.cpp", tmp_path / "index"
    src.write_text(SOURCE)
    include = build._nvcc().rsplit("/bin/", 1)[0] + "/include"
    subprocess.run(["g++", "-std=c++17", "-I", include, "-I", build.CSRC, "-o", str(exe), str(src)],
                   check=True)
    out = subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout.split()
    assert out == [str(2 * (2**31 - 1)), str(2 * (2**31 - 1) - 3), "300", str(300 * 299 // 2)]
