"""The bounded wait between warps of a diagonal block's leaf: a flag that nothing sets ends the wait and is reported."""
import ctypes
import os
import subprocess

import pytest

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "tc_common.cuh"
using namespace exa;
// one warp; flag 0 is set to 5 before the waits, flag 1 never; out: timeout, site, polls left for each flag
__global__ void waits(DevStatus* st, int* out, int limit) {
  __shared__ int flag[2];
  if (threadIdx.x < 2) flag[threadIdx.x] = 0;
  __syncthreads();
  if (threadIdx.x == 0) tc::post(flag, 5);
  __syncthreads();
  int polls = limit;
  tc::await(flag, 5, polls);
  tc::report_waits(polls, st, 7);
  if (threadIdx.x == 0) { out[0] = st->timeout; out[1] = polls; }
  __syncthreads();
  tc::await(flag + 1, 5, polls);
  tc::report_waits(polls, st, 8);
  __syncthreads();
  if (threadIdx.x == 0) { out[2] = st->timeout; out[3] = st->timeout_where; out[4] = polls; }
  tc::await(flag + 1, 5, polls);  // at once
}
extern "C" int run(int limit, int* out) {
  DevStatus* st;
  int* d;
  if (cudaMalloc(&st, sizeof(DevStatus)) != cudaSuccess || cudaMalloc(&d, 32) != cudaSuccess) return 1;
  cudaMemset(st, 0, sizeof(DevStatus));
  waits<<<1, 32>>>(st, d, limit);
  int rc = cudaMemcpy(out, d, 5 * sizeof(int), cudaMemcpyDeviceToHost) != cudaSuccess;
  cudaFree(st);
  cudaFree(d);
  return rc;
}
"""


def test_a_wait_that_runs_out_is_reported(tmp_path):
    from paper_1908_06936_gb300 import build

    src, so = tmp_path / "waits.cu", tmp_path / "waits.so"
    src.write_text(SOURCE)
    subprocess.check_call([build._nvcc()] + build.ARCH + build.NVCC_FLAGS + ["-I" + build.CSRC, "-shared", "-o", str(so),
                                                                            str(src)])
    out = (ctypes.c_int * 5)()
    assert ctypes.CDLL(os.fspath(so)).run(1 << 12, out) == 0
    assert out[0] == 0 and out[1] > 0          # the flag that is set
    assert (out[2], out[3]) == (1, 8) and out[4] <= 0
