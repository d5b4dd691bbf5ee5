"""Shared-memory limits are raised once per kernel and device (the CUDA calls
replaced by host functions that record their arguments)."""

import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2301_09889_gb300", "csrc")

SOURCE = r"""
#include "smem_limit.h"
#include <cstdio>
static int device = 0, limit[2] = {48 << 10, 48 << 10}, calls = 0;
extern "C" cudaError_t cudaGetDevice(int* d) { *d = device; return cudaSuccess; }
extern "C" cudaError_t cudaFuncSetAttribute(const void*, cudaFuncAttribute a, int v) {
  ++calls;
  if (a == cudaFuncAttributeMaxDynamicSharedMemorySize) limit[device] = v;
  return cudaSuccess;
}
static void kernel() {}
int main() {
  chdns::SmemLimit lim;
  const int sizes[] = {52 << 10, 40 << 10, 60 << 10, 60 << 10};
  for (int size : sizes)
    for (device = 0; device < 2; ++device)
      if (chdns::raise_smem_limit(kernel, &lim, size) != cudaSuccess || limit[device] < size) {
        std::printf("device %d below %d\n", device, size);
        return 1;
      }
  std::printf("%d\n", calls);
  return calls == 4 && limit[0] == 60 << 10 && limit[1] == 60 << 10 ? 0 : 1;
}
"""


def test_limits_are_kept_per_device(tmp_path):
    include = "/usr/local/cuda/include"
    gxx = shutil.which("g++")
    if not gxx or not os.path.exists(os.path.join(include, "cuda_runtime_api.h")):
        pytest.skip("no host compiler or CUDA headers")
    src = tmp_path / "limits.cpp"
    src.write_text(SOURCE)
    exe = tmp_path / "limits"
    subprocess.run([gxx, "-std=c++17", "-I", CSRC, "-I", include, str(src), "-o", str(exe), "-pthread"], check=True)
    run = subprocess.run([str(exe)], capture_output=True, text=True)
    assert run.returncode == 0, run.stdout
