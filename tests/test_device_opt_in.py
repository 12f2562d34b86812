"""The opt-in of a kernel to large dynamic shared memory belongs to the device that
is current: made once on each, by whichever thread comes first, and not remembered
when it failed.  Against a fake runtime of two devices, so that no GPU is needed."""
import os
import shutil
import subprocess

import pytest

from paper_2607_20791_gb300.build import CSRC, INCLUDE

SOURCE = r"""
#include <cstdlib>
#include <thread>
#include <vector>
#include "common.h"
static thread_local int g_dev = 0;
static std::atomic<int> g_calls[2];
static std::atomic<bool> g_fail{false};
extern "C" cudaError_t cudaGetDevice(int* d) { *d = g_dev; return cudaSuccess; }
extern "C" cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute, int) {
  if (g_fail) return cudaErrorInvalidValue;
  ++g_calls[g_dev];
  return cudaSuccess;
}
extern "C" const char* cudaGetErrorString(cudaError_t) { return "fake"; }
int rgd::set_error(int code, const char*, ...) { return code; }
#define CHECK(x) if (!(x)) { printf("line %d: %s\n", __LINE__, #x); return 1; }
int main() {
  static std::atomic<bool> done[rgd::kMaxDevices] = {}, other[rgd::kMaxDevices] = {};
  const void* kernel = &g_fail;
  g_fail = true;
  CHECK(rgd::ensure_smem(kernel, 100000, done) == RGD_ERR_CUDA);
  g_fail = false;
  for (int i = 0; i < 3; ++i)
    for (g_dev = 0; g_dev < 2; ++g_dev) CHECK(rgd::ensure_smem(kernel, 100000, done) == RGD_OK);
  CHECK(g_calls[0] == 1 && g_calls[1] == 1);  // each device, once
  std::vector<std::thread> t;
  for (int i = 0; i < 8; ++i)
    t.emplace_back([kernel, i] {
      g_dev = i & 1;
      if (rgd::ensure_smem(kernel, 100000, other) != RGD_OK || !other[g_dev]) abort();
    });
  for (auto& x : t) x.join();
  CHECK(g_calls[0] >= 2 && g_calls[1] >= 2);
  return 0;
}
"""


def test_opt_in_once_per_device(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    inc = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")
    if not os.path.exists(os.path.join(inc, "cuda_runtime.h")) or not shutil.which("g++"):
        pytest.skip("no CUDA headers or no g++")
    src, exe = tmp_path / "opt_in.cpp", tmp_path / "opt_in"
    src.write_text(SOURCE)
    res = subprocess.run(["g++", "-std=c++17", "-pthread", "-I", CSRC, "-I", INCLUDE, "-I", inc, str(src), "-o", str(exe)],
                         capture_output=True, text=True)
    assert res.returncode == 0, res.stderr
    res = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert res.returncode == 0, res.stdout
