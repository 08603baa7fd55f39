"""The look-ahead stream is joined to the main one wherever a factorisation returns (host code, on a recorded CUDA API)."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1908_06936_gb300", "csrc")

SOURCE = r"""
#include <cstdio>
#include "side_join.cuh"
// streams 1 (main) and 2 (side), events 3 (fork) and 4 (side's end)
static int id(const void* p) { return (int)(size_t)p; }
extern "C" cudaError_t cudaEventRecord(cudaEvent_t e, cudaStream_t s) {
  std::printf("record %d on %d;", id(e), id(s));
  return cudaSuccess;
}
extern "C" cudaError_t cudaStreamWaitEvent(cudaStream_t s, cudaEvent_t e, unsigned int) {
  std::printf("%d waits %d;", id(s), id(e));
  return cudaSuccess;
}
static void factor(int stop) {  // two steps; returns early at `stop`
  const cudaEvent_t ev[2] = {(cudaEvent_t)3, (cudaEvent_t)4};
  exa::SideJoin j((cudaStream_t)1, (cudaStream_t)2, ev);
  for (int k = 0; k < 2; ++k) {
    if (stop == 10 * k) return;
    j.fork();
    if (stop == 10 * k + 1) return;
    j.side_done();
    if (stop == 10 * k + 2) return;
    j.join();
  }
}
int main() {
  for (int stop : {0, 1, 2, 10, 11, 12, 99}) {
    std::printf("%d:", stop);
    factor(stop);
    std::printf("\n");
  }
}
"""


def test_every_fork_is_joined(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    inc = "/usr/local/cuda/include"
    if not cxx or not os.path.exists(os.path.join(inc, "cuda_runtime_api.h")):
        pytest.skip("no C++ compiler or CUDA headers")
    (tmp_path / "join.cpp").write_text(SOURCE.replace("#include <cstdio>", "#include <cstdio>\n#include <initializer_list>"))
    subprocess.check_call([cxx, "-std=c++17", "-I" + CSRC, "-I" + inc, "-o", str(tmp_path / "join"), str(tmp_path / "join.cpp")])
    out = dict(l.split(":") for l in subprocess.check_output([str(tmp_path / "join")], text=True).splitlines())
    step = "record 3 on 1;2 waits 3;record 4 on 2;1 waits 4;"
    assert out == {"0": "", "1": step, "2": step, "10": step, "11": step * 2, "12": step * 2, "99": step * 2}
