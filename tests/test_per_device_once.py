"""Settings that belong to a device (a kernel's shared-memory limit) are made on
every device of the process, once, also when threads race for it, and again
after a failure.  Compiled for the host with a stand-in for cudaGetDevice."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2307_04508_gb300", "csrc")

SRC = r"""
#include "per_device.h"
#include <stdio.h>
#include <thread>
#include <vector>
static thread_local int g_dev = 0;
extern "C" cudaError_t cudaGetDevice(int *d) { *d = g_dev; return cudaSuccess; }
int main() {
  ltgw::OncePerDevice once;
  std::atomic<int> calls[3] = {};
  std::vector<std::thread> ts;
  for (int t = 0; t < 12; ++t)
    ts.emplace_back([&, t] {
      g_dev = t % 3;
      for (int i = 0; i < 1000; ++i)
        if (once([&] { ++calls[g_dev]; return cudaSuccess; }) != cudaSuccess) ++calls[0];
    });
  for (auto &t : ts) t.join();
  ltgw::OncePerDevice retry;
  int tries = 0;
  const cudaError_t a = retry([&] { ++tries; return cudaErrorMemoryAllocation; });
  const cudaError_t b = retry([&] { ++tries; return cudaSuccess; });
  const cudaError_t c = retry([&] { ++tries; return cudaErrorMemoryAllocation; });
  printf("%d %d %d %d %d %d %d\n", (int)calls[0], (int)calls[1], (int)calls[2], tries,
         a == cudaErrorMemoryAllocation, b == cudaSuccess, c == cudaSuccess);
}
"""


def test_once_on_each_device(tmp_path):
    from paper_2307_04508_gb300 import build
    src, exe = tmp_path / "once.cpp", tmp_path / "once"
    src.write_text(SRC)
    inc = os.path.join(os.path.dirname(os.path.dirname(build.nvcc())), "include")
    subprocess.check_call(["g++", "-std=c++17", "-pthread", "-I", CSRC, "-I", inc, str(src), "-o", str(exe)])
    assert subprocess.check_output([str(exe)], text=True).split() == ["1", "1", "1", "2", "1", "1", "1"]


def test_no_process_wide_guard_of_a_kernel_attribute():
    for f in sorted(os.listdir(CSRC)):
        text = open(os.path.join(CSRC, f)).read()
        for block in text.split("std::call_once(")[1:]:
            assert "cudaFuncSetAttribute" not in block.split("});")[0], f
