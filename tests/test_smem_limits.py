"""The limit of a kernel's dynamic shared memory (csrc/vrm_smem.cuh) belongs to
kernel and device: set once on every device that launches the kernel, again
after a failure, and by several threads at once to one value.  Compiled here
against stand-ins for the three runtime calls."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CUDA = os.environ.get("CUDA_HOME", "/usr/local/cuda")

SOURCE = r"""
#include <cstdio>
#include <map>
#include <mutex>
#include <thread>
#include <vector>
#include "vrm_smem.cuh"

static std::mutex mu;
static std::map<std::pair<const void*, int>, std::vector<int>> sets;  // (kernel, device): values
static thread_local int device = 0;
static cudaError_t next_error = cudaSuccess;
extern "C" cudaError_t cudaGetDevice(int* d) { *d = device; return cudaSuccess; }
extern "C" cudaError_t cudaFuncSetAttribute(const void* f, cudaFuncAttribute a, int v) {
  std::lock_guard<std::mutex> l(mu);
  if (a != cudaFuncAttributeMaxDynamicSharedMemorySize) return cudaErrorInvalidValue;
  if (next_error != cudaSuccess) return next_error;
  sets[{f, device}].push_back(v);
  return cudaSuccess;
}
void one(int) {}
void two(int) {}
template <int K> void many(int) {}
#define CHECK(c) do { if (!(c)) { std::printf("line %d: %s\n", __LINE__, #c); return 1; } } while (0)
int main() {
  using vrm::allow_smem;
  const void *p1 = (const void*)&one, *p2 = (const void*)&two;
  CHECK(allow_smem<one>(100) == cudaSuccess && allow_smem<one>(100) == cudaSuccess);
  CHECK((sets[{p1, 0}] == std::vector<int>{100}));
  device = 1;  // another device has a limit of its own
  CHECK(allow_smem<one>(100) == cudaSuccess && allow_smem<one>(100) == cudaSuccess);
  CHECK((sets[{p1, 1}] == std::vector<int>{100}) && sets[std::make_pair(p1, 0)].size() == 1);
  // and so has another kernel; a failure is reported and tried again
  next_error = cudaErrorInvalidValue;
  CHECK(allow_smem<two>(200) == cudaErrorInvalidValue);
  next_error = cudaSuccess;
  CHECK(allow_smem<two>(200) == cudaSuccess);
  CHECK((sets[{p2, 1}] == std::vector<int>{200}) && (sets.count({p2, 0}) == 0));
  device = 64;  // beyond the devices that are kept: set every time
  CHECK(allow_smem<two>(200) == cudaSuccess && allow_smem<two>(200) == cudaSuccess);
  CHECK((sets[{p2, 64}] == std::vector<int>{200, 200}));
  std::vector<std::thread> t;
  for (int k = 0; k < 16; ++k)
    t.emplace_back([k] {
      device = k % 4;
      for (int r = 0; r < 100; ++r) allow_smem<many<7>>(300);
    });
  for (auto& x : t) x.join();
  for (int d = 0; d < 4; ++d) {
    const auto& v = sets[{(const void*)&many<7>, d}];
    CHECK(v.size() >= 1 && v.size() <= 4);  // at most once by each of a device's threads
    for (int b : v) CHECK(b == 300);
  }
  return 0;
}
"""


def test_limit_is_set_once_per_kernel_and_device(tmp_path):
    cxx = shutil.which("g++")
    if not cxx or not os.path.exists(os.path.join(CUDA, "include", "cuda_runtime_api.h")):
        pytest.skip("no C++ compiler or CUDA headers")
    src, exe = tmp_path / "smem.cpp", tmp_path / "smem"
    src.write_text(SOURCE)
    subprocess.run([cxx, "-std=c++17", "-O1", "-pthread", "-I", os.path.join(CUDA, "include"), "-I",
                    os.path.join(ROOT, "paper_1508_06379_gb300", "csrc"), str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout


def test_every_limit_goes_through_it():
    d = os.path.join(ROOT, "paper_1508_06379_gb300", "csrc")
    for name in sorted(os.listdir(d)):
        if name != "vrm_smem.cuh":
            assert "cudaFuncSetAttribute" not in open(os.path.join(d, name)).read(), name
