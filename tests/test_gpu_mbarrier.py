"""The layer's mbarrier wait (csrc/mbarrier.cuh): a phase that completes ends
it, and one that never does ends it by the clock, with a status that the host
reads and the context still usable."""
import ctypes
import os
import subprocess

import pytest
import torch

from paper_2601_01473_gb300 import build

pytestmark = pytest.mark.gpu

# One warp waits for a phase with n_arrive of its two arrivals; result[0] = how
# the wait ended, result[1] = its nanoseconds.
SOURCE = r"""
#include "mbarrier.cuh"
using namespace agnes;
__global__ void wait_kernel(int n_arrive, unsigned long long* result) {
  __shared__ uint64_t bar;
  const uint32_t b = (uint32_t)__cvta_generic_to_shared(&bar);
  if (threadIdx.x == 0) mbar_init(b, 2);
  __syncthreads();
  if (threadIdx.x >= 32 && (int)threadIdx.x < 32 + n_arrive) mbar_arrive(b);
  if (threadIdx.x < 32) {
    const uint64_t t = global_ns();
    const bool ok = mbar_wait(b, 0);
    if (threadIdx.x == 0) {
      result[0] = ok ? 1 : 2;
      result[1] = global_ns() - t;
    }
  }
}
extern "C" int run(int n_arrive, unsigned long long* host) {
  unsigned long long* d = nullptr;
  if (cudaMalloc(&d, 16) != cudaSuccess) return 1;
  wait_kernel<<<1, 64>>>(n_arrive, d);
  const cudaError_t e = cudaMemcpy(host, d, 16, cudaMemcpyDeviceToHost);
  cudaFree(d);
  return e != cudaSuccess;
}
"""


def test_a_wait_ends_by_arrival_or_by_the_clock(cuda_device, tmp_path):
    src, so = tmp_path / "wait.cu", tmp_path / "libwait.so"
    src.write_text(SOURCE)
    subprocess.run([build._nvcc(), *build.ARCH, *build.NVCC_FLAGS, "-I", build.CSRC, "-shared",
                    "-cudart", "static", "-o", str(so), str(src)], check=True)
    run = ctypes.CDLL(os.fspath(so)).run
    out = (ctypes.c_ulonglong * 2)()
    for n_arrive, ended in ((2, 1), (1, 2), (2, 1)):
        assert run(n_arrive, out) == 0
        assert out[0] == ended
        if ended == 2:
            assert 1e9 <= out[1] < 1.5e9, out[1]
        else:
            assert out[1] < 1e8, out[1]
    assert float(torch.ones(8, device=cuda_device).sum()) == 8.0
