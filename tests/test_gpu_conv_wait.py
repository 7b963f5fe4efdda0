"""The bounded wait of the convolution kernels (csrc/nn_wait.cuh): a phase that completes is seen, one that nothing
completes ends in about two seconds with a status, and the device goes on."""
import os
import subprocess

import pytest

from paper_2311_05091_gb300.build import ARCH, CSRC, nvcc

pytestmark = pytest.mark.gpu

PROBE = r"""
#include <cstdio>
#include <cuda_runtime.h>
#include "nn_wait.cuh"
using namespace lbm_nn;
// one warp, two barriers: lane 0 arrives on the first; nothing arrives on the second
__device__ unsigned long long now() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
__global__ void probe(int* seen, unsigned long long* ns) {
  __shared__ unsigned long long bar[2];
  const uint32_t b = (uint32_t)__cvta_generic_to_shared(bar);
  if (threadIdx.x == 0) {
    mbar_init(b, 1);
    mbar_init(b + 8, 1);
  }
  __syncthreads();
  if (threadIdx.x == 0) mbar_arrive(b);
  for (int k = 0; k < 2; ++k) {
    const unsigned long long t = now();
    const bool ok = mbar_wait(b + 8 * k, 0);
    if (threadIdx.x == 0) seen[k] = ok, ns[k] = now() - t;
  }
}
int main() {
  int* seen;
  unsigned long long* ns;
  if (cudaMallocManaged(&seen, 8) != cudaSuccess || cudaMallocManaged(&ns, 16) != cudaSuccess) return 1;
  probe<<<1, 32>>>(seen, ns);
  if (cudaDeviceSynchronize() != cudaSuccess) return 2;
  printf("%d %d %g %g\n", seen[0], seen[1], ns[0] * 1e-9, ns[1] * 1e-9);
  return 0;
}
"""


def test_a_wait_ends_with_a_status(tmp_path):
    src, exe = tmp_path / "probe.cu", tmp_path / "probe"
    src.write_text(PROBE)
    subprocess.run([nvcc(), *ARCH, "-std=c++17", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True, timeout=60).stdout.split()
    assert out[:2] == ["1", "0"]
    assert float(out[2]) < 0.1 and 1.9 < float(out[3]) < 3.0
