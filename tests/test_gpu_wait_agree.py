"""Threads whose bounded waits end differently agree on the outcome and leave together.

A program of its own, on csrc/jf_device.cuh: of 256 threads half wait on an mbarrier that nothing arrives at
(5 ms limit) and half, lane by lane, on one that is complete. All must come out of sync_and with "gave up"; in
a second round, where every wait succeeds, with "ready". Nothing else is in flight.
"""
import os
import subprocess

import pytest

from paper_2512_14681_gb300 import build as B
from tests.parity import need_gpu

pytestmark = pytest.mark.gpu

PROGRAM = r"""
#include <cstdio>
#include "jf_device.cuh"
__global__ void k_agree(int* out) {
  __shared__ __align__(8) uint64_t done, never;
  if (threadIdx.x == 0) {
    mbar_init(smem_u32(&done), 1);
    mbar_init(smem_u32(&never), 1);
    fence_mbar_init();
    mbar_arrive(smem_u32(&done));
  }
  __syncthreads();
  const bool waits_long = (threadIdx.x ^ (threadIdx.x >> 5)) & 1;
  const bool own = mbar_wait_bounded(smem_u32(waits_long ? &never : &done), 0u, 5000000ull);
  const bool all = sync_and<3, 256>(own);
  const bool again = sync_and<3, 256>(mbar_wait_bounded(smem_u32(&done), 0u, 5000000ull));
  atomicAdd(out, own == !waits_long);
  atomicAdd(out + 1, !all);
  atomicAdd(out + 2, again);
}
int main() {
  int* d;
  int h[3] = {};
  if (cudaMalloc(&d, sizeof(h)) || cudaMemset(d, 0, sizeof(h))) return 1;
  k_agree<<<1, 256>>>(d);
  if (cudaMemcpy(h, d, sizeof(h), cudaMemcpyDeviceToHost)) return 1;
  std::printf("%d %d %d\n", h[0], h[1], h[2]);
}
"""


def test_threads_leave_together(tmp_path):
    need_gpu()
    src, exe = tmp_path / "agree.cu", tmp_path / "agree"
    src.write_text(PROGRAM)
    r = subprocess.run([B.nvcc(), *B.ARCH, "-std=c++17", "--expt-relaxed-constexpr", "-I", B.CSRC, str(src), "-o", str(exe)],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    out = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert out.returncode == 0 and out.stdout.split() == ["256", "256", "256"]
