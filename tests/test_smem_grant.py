"""Shared-memory limits of kernels, on the CPU: smem_grant.h with a fake of the
driver's call.  The limit is a single value that every call overwrites, so a
launch that needs little must not lower what a launch on another thread has just
been granted; each device has its own limit; a refusal is passed on and tried
again.
"""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2010_15069_gb300", "csrc")

CHECK = r"""
#include <chrono>
#include <cstdio>
#include <thread>
#include <vector>
#include "smem_grant.h"
using spgpe::SmemGrant;

std::atomic<size_t> limit[SmemGrant::kDevices];  // what the driver holds
std::atomic<int> calls;
cudaError_t fake(int dev, size_t b) {
  ++calls;
  std::this_thread::sleep_for(std::chrono::microseconds(200));
  limit[dev] = b;
  return cudaSuccess;
}

int main() {
  int bad = 0;
  for (int round = 0; round < 20; ++round) {
    SmemGrant g;
    for (auto &l : limit) l = 48 * 1024;
    std::vector<std::thread> th;
    for (int t = 0; t < 8; ++t)
      th.emplace_back([&, t] {
        for (int i = 0; i < 8; ++i) {
          const int dev = t & 1;
          const size_t need = 1024 * (50 + (37 * (t + 3 * i + round)) % 170);
          if (g.raise(dev, need, [&](size_t b) { return fake(dev, b); }) != cudaSuccess) ++bad;
          if (limit[dev] < need) ++bad;  // the launch would be refused
        }
      });
    for (auto &t : th) t.join();
  }
  printf("lowered %d\n", bad);
  SmemGrant g;
  calls = 0;
  int refused = 0;
  auto no = [&](size_t) { ++refused; return cudaErrorInvalidValue; };
  printf("refusal %d %d\n", g.raise(0, 300000, no) == cudaErrorInvalidValue, g.raise(0, 300000, no) == cudaErrorInvalidValue);
  g.raise(0, 100000, [&](size_t b) { return fake(0, b); });
  g.raise(0, 60000, [&](size_t b) { return fake(0, b); });
  g.raise(1, 60000, [&](size_t b) { return fake(1, b); });
  printf("calls %d refused %d limits %zu %zu\n", (int)calls, refused, (size_t)limit[0], (size_t)limit[1]);
  printf("device %d %d\n", g.raise(-1, 1, no) == cudaErrorInvalidDevice, g.raise(64, 1, no) == cudaErrorInvalidDevice);
  return 0;
}
"""


def test_limits_are_only_raised_per_device(tmp_path):
    nvcc = next((c for c in (shutil.which("nvcc"), "/usr/local/cuda/bin/nvcc") if c and os.path.exists(c)), None)
    if nvcc is None:
        pytest.skip("nvcc not found")
    src, exe = tmp_path / "check.cu", tmp_path / "check"
    src.write_text(CHECK)
    subprocess.run([nvcc, "-std=c++17", "-gencode", "arch=compute_103a,code=sm_103a", "-I", CSRC, str(src), "-o",
                    str(exe)], check=True, timeout=900)
    out = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60, check=True).stdout.split("\n")
    assert out[:4] == ["lowered 0", "refusal 1 1", "calls 2 refused 2 limits 100000 60000", "device 1 1"], out
