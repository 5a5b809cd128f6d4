"""The shared-memory limit of a kernel belongs to a device: it is set on each one
that launches the kernel, and threads that launch at once agree on it. The
library's helper, compiled against stand-ins of the two runtime calls."""
import glob
import os
import re
import shutil
import subprocess

import pytest

from paper_2609_34867_gb300 import build as B

PROGRAM = r"""
#include "p4q_smem_limit.h"
#include <cassert>
#include <map>
#include <mutex>
#include <thread>
#include <vector>

static thread_local int device = 0;
static std::mutex mu;
static std::map<std::pair<int, const void*>, std::vector<int>> set;  // (device, kernel) -> the sizes set
static cudaError_t answer = cudaSuccess;

extern "C" cudaError_t cudaGetDevice(int* d) { *d = device; return cudaSuccess; }
extern "C" cudaError_t cudaFuncSetAttribute(const void* f, cudaFuncAttribute a, int bytes) {
  assert(a == cudaFuncAttributeMaxDynamicSharedMemorySize);
  std::lock_guard<std::mutex> l(mu);
  if (answer == cudaSuccess) set[{device, f}].push_back(bytes);
  return answer;
}
void kernel(int) {}

int main() {
  const void* k = reinterpret_cast<const void*>(&kernel);
  p4q::SmemLimit one;
  answer = cudaErrorInvalidValue;  // a failure is reported and not remembered
  assert(one.allow(kernel, 100000) == cudaErrorInvalidValue);
  answer = cudaSuccess;
  for (int i = 0; i < 3; ++i) assert(one.allow(kernel, 100000) == cudaSuccess);
  assert((set.size() == 1 && set[{0, k}] == std::vector<int>{100000}));
  device = 1;  // another device of the process
  for (int i = 0; i < 3; ++i) assert(one.allow(kernel, 100000) == cudaSuccess);
  assert((set.size() == 2 && set[{1, k}] == std::vector<int>{100000}));
  device = 70;  // past the devices it keeps: set each time
  for (int i = 0; i < 3; ++i) assert(one.allow(kernel, 100000) == cudaSuccess);
  assert((set[{70, k}].size() == 3));
  set.clear();
  p4q::SmemLimit many;
  std::vector<std::thread> ts;
  for (int t = 0; t < 16; ++t)
    ts.emplace_back([&, t] {
      device = t % 4;
      for (int i = 0; i < 1000; ++i) assert(many.allow(kernel, 232192) == cudaSuccess);
    });
  for (auto& t : ts) t.join();
  assert(set.size() == 4);
  for (auto& s : set)
    for (int bytes : s.second) assert(bytes == 232192);
  return 0;
}
"""


def test_limit_per_device_and_thread(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    src, exe = tmp_path / "limit.cpp", tmp_path / "limit"
    src.write_text(PROGRAM)
    inc = os.path.join(os.path.dirname(os.path.dirname(B.nvcc())), "include")
    subprocess.run([cxx, "-std=c++17", "-O1", "-UNDEBUG", "-pthread", "-I", B.CSRC, "-isystem", inc, str(src), "-o",
                    str(exe)], check=True)
    subprocess.run([str(exe)], check=True, timeout=60)


def test_no_launch_keeps_the_limit_by_itself():
    """Every launch sets the limit through the helper (or on each call), to a
    fixed size and not to that of the call."""
    for path in sorted(glob.glob(os.path.join(B.CSRC, "*.cu"))):
        code = re.sub(r"//[^\n]*", "", open(path).read())
        assert "static bool attr_set" not in code and "smem_set" not in code, path
        sizes = re.findall(r"cudaFuncSetAttribute\([^;]*?,\s*cudaFuncAttributeMaxDynamicSharedMemorySize,\s*([^;]*)\);", code)
        assert sizes == (["static_cast<int>(kDivSmem)"] if path.endswith("p4q_diverse.cu") else []), path
