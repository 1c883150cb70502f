"""Kernels that ask for more than the default dynamic shared memory, on several devices and threads of one process
(no GPU): the limit is an attribute of a kernel on one device.  csrc/mw_smem.h is compiled against a stand-in for the
two CUDA runtime calls that it makes; no launcher sets the attribute another way."""
import os
import shutil
import subprocess

import pytest

from paper_2311_05322_gb300 import build

HARNESS = r"""
#include "mw_smem.h"
#include <cassert>
#include <cstdio>
#include <map>
#include <mutex>
#include <thread>
#include <vector>
static thread_local int current = 0;
static std::mutex mu;
static std::map<std::pair<int, const void*>, int> value;
static int calls = 0, fail_next = 0;
extern "C" cudaError_t cudaGetDevice(int* d) { *d = current; return cudaSuccess; }
extern "C" cudaError_t cudaFuncSetAttribute(const void* f, cudaFuncAttribute a, int v) {
  std::lock_guard<std::mutex> lock(mu);
  assert(a == cudaFuncAttributeMaxDynamicSharedMemorySize);
  ++calls;
  if (fail_next > 0) { --fail_next; return cudaErrorInvalidValue; }
  value[{current, f}] = v;
  return cudaSuccess;
}
void kernel_a(int) {}
void kernel_b(float) {}
int main() {
  mwk::SmemLimit a, b;
  for (int round = 0; round < 2; ++round)
    for (current = 0; current < 3; ++current) {
      a.raise(kernel_a, 100000);
      assert(value.at({current, (const void*)kernel_a}) == 100000);
    }
  assert(calls == 3);                      // once per device
  current = 2;
  fail_next = 1;
  b.raise(kernel_b, 60000);                // refused: tried again at the next launch
  b.raise(kernel_b, 60000);
  b.raise(kernel_b, 60000);
  assert(calls == 5 && value.at({2, (const void*)kernel_b}) == 60000);
  current = 70;                            // beyond the remembered devices: at every launch
  b.raise(kernel_b, 60000);
  b.raise(kernel_b, 60000);
  assert(calls == 7 && value.at({70, (const void*)kernel_b}) == 60000);
  mwk::SmemLimit c;
  std::vector<std::thread> ts;
  for (int t = 0; t < 16; ++t)
    ts.emplace_back([&c, t] {
      current = t % 4;
      for (int i = 0; i < 100; ++i) {
        c.raise(kernel_b, 70000);
        std::lock_guard<std::mutex> lock(mu);
        assert(value.at({current, (const void*)kernel_b}) == 70000);
      }
    });
  for (auto& t : ts) t.join();
  puts("ok");
}
"""


def test_once_per_kernel_and_device(tmp_path):
    include = os.path.join(os.path.dirname(os.path.dirname(build.nvcc())), "include")
    if shutil.which("g++") is None:
        pytest.skip("no g++")
    src, exe = tmp_path / "harness.cpp", tmp_path / "harness"
    src.write_text(HARNESS)
    subprocess.run(["g++", "-std=c++17", "-O1", "-UNDEBUG", "-I", build.CSRC, "-isystem", include, str(src), "-o",
                    str(exe), "-pthread"], check=True)
    assert subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout == "ok\n"


def test_no_launcher_sets_it_another_way():
    for name in sorted(os.listdir(build.CSRC)):
        with open(os.path.join(build.CSRC, name)) as f:
            if "cudaFuncSetAttribute" in f.read():
                assert name == "mw_smem.h", name
