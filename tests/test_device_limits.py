"""Per-device launch state (csrc/smem_limit.cuh) against a stand-in for the CUDA runtime, on the CPU.

The header is compiled into a host program whose cudaGetDevice,
cudaFuncSetAttribute and cudaDeviceGetAttribute are fakes that keep a limit per
(kernel, device), as the runtime does.
"""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

RUNTIME = r"""
#pragma once
#include <cstddef>
enum cudaError_t { cudaSuccess = 0, cudaErrorInvalidValue = 1 };
enum { cudaFuncAttributeMaxDynamicSharedMemorySize = 8, cudaDevAttrMultiProcessorCount = 16 };
extern thread_local int fake_device;
extern int fake_calls;
cudaError_t fake_set(const void *kernel, int bytes);
inline cudaError_t cudaGetDevice(int *d) { *d = fake_device; return cudaSuccess; }
template <class K> cudaError_t cudaFuncSetAttribute(K *k, int, int bytes) { return fake_set((const void *)k, bytes); }
inline cudaError_t cudaDeviceGetAttribute(int *v, int, int dev) { *v = 100 + dev; return cudaSuccess; }
"""

PROGRAM = r"""
#include <cstdio>
#include <map>
#include <thread>
#include <utility>
#include <vector>
#include "smem_limit.cuh"
thread_local int fake_device = 0;
int fake_calls = 0;
static std::map<std::pair<const void *, int>, int> limits;
cudaError_t fake_set(const void *kernel, int bytes) {
  ++fake_calls;
  if (bytes > 232448) return cudaErrorInvalidValue;
  limits[{kernel, fake_device}] = bytes;
  return cudaSuccess;
}
static void kernel() {}
#define CHECK(x) if (!(x)) { std::printf("line %d: %s\n", __LINE__, #x); return 1; }
int main() {
  static mra::SmemLimit granted;
  auto raise = [&](int dev, size_t bytes) { fake_device = dev; return mra::raise_smem_limit(kernel, bytes, granted); };
  auto limit = [&](int dev) { return limits[{(const void *)kernel, dev}]; };
  for (int dev : {0, 1, 63, 64, 100}) {  // every device gets its own limit
    CHECK(raise(dev, 100000) == cudaSuccess && limit(dev) == 100000);
    CHECK(raise(dev, 200000) == cudaSuccess && limit(dev) == 200000);
  }
  const int calls = fake_calls;
  CHECK(raise(0, 50000) == cudaSuccess && raise(63, 200000) == cudaSuccess);
  CHECK(limit(0) == 200000 && limit(63) == 200000 && fake_calls == calls);  // never lowered, not set again
  CHECK(raise(2, 300000) != cudaSuccess && raise(2, 100000) == cudaSuccess && limit(2) == 100000);
  std::vector<std::thread> threads;
  bool ok[16] = {};
  for (int i = 0; i < 16; ++i)
    threads.emplace_back([&ok, i] {
      fake_device = i % 8 == 7 ? 70 : i % 8;
      bool all = true;
      for (int j = 0; j < 1000; ++j) {
        int n = 0;
        all = all && mra::sm_count(&n) == cudaSuccess && n == 100 + fake_device;
      }
      ok[i] = all;
    });
  for (auto &t : threads) t.join();
  for (bool o : ok) CHECK(o);
  return 0;
}
"""


def test_limits_and_sm_counts_are_kept_per_device(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no C++ compiler")
    (tmp_path / "cuda_runtime.h").write_text(RUNTIME)
    (tmp_path / "t.cpp").write_text(PROGRAM)
    exe = tmp_path / "t"
    r = subprocess.run([cxx, "-std=c++17", "-O1", "-pthread", "-I", str(tmp_path),
                        "-I", os.path.join(ROOT, "paper_2011_05755_gb300", "csrc"), str(tmp_path / "t.cpp"),
                        "-o", str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout


def test_every_launcher_uses_the_per_device_record():
    csrc = os.path.join(ROOT, "paper_2011_05755_gb300", "csrc")
    for f in sorted(os.listdir(csrc)):
        text = open(os.path.join(csrc, f)).read()
        assert f == "smem_limit.cuh" or "cudaFuncSetAttribute(" not in text, f
