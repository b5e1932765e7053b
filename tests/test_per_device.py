"""Kernel settings made once per device, against a stand-in for the CUDA
runtime's two calls: a second device, a setting that fails, several threads."""
import glob
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2403_09010_gb300", "csrc")

PROGRAM = r"""
#include <stdio.h>
#include <atomic>
#include <thread>
#include <vector>
#include "per_device.h"
static thread_local int t_device = 0;
static std::atomic<int> g_limits[65][2];  // by device and kernel
static std::atomic<int> g_fail{0};
extern "C" cudaError_t cudaGetDevice(int* d) { *d = t_device; return cudaSuccess; }
extern "C" cudaError_t cudaFuncSetAttribute(const void* f, cudaFuncAttribute, int) {
  if (g_fail > 0) { --g_fail; return cudaErrorInvalidValue; }
  ++g_limits[t_device][f ? 1 : 0];
  return cudaSuccess;
}
static int k;
template <int N>
void launch() {  // as the launchers do it, a static object each
  static xtn::PerDevice shared;
  shared([] { return xtn::allow_shared(N ? &k : nullptr, 1 << 17, N != 0); });
}
#define CHECK(x) do { if (!(x)) { printf("line %d: %s\n", __LINE__, #x); return 1; } } while (0)
int main() {
  for (int dev : {0, 1, 0, 5, 1, 63}) { t_device = dev; launch<1>(); launch<0>(); }
  for (int dev : {0, 1, 5, 63}) CHECK(g_limits[dev][1] == 2 && g_limits[dev][0] == 1);
  CHECK(g_limits[2][0] == 0 && g_limits[2][1] == 0);
  t_device = 2;
  g_fail = 1;
  launch<1>();  // refused: the next call sets it
  CHECK(g_limits[2][1] == 0);
  launch<1>(); launch<1>();
  CHECK(g_limits[2][1] == 2);
  t_device = 64;  // more than it keeps note of: set every time
  launch<1>(); launch<1>();
  CHECK(g_limits[64][1] == 4);
  std::vector<std::thread> all;
  for (int i = 0; i < 8; ++i)
    all.emplace_back([i] { t_device = 10 + i % 4; for (int r = 0; r < 100; ++r) launch<1>(); });
  for (auto& t : all) t.join();
  for (int dev = 10; dev < 14; ++dev) CHECK(g_limits[dev][1] >= 2 && g_limits[dev][1] <= 4);
  return 0;
}
"""


def test_set_on_every_device(tmp_path):
    cuda = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    gxx = shutil.which("g++")
    if not gxx or not os.path.exists(os.path.join(cuda, "include", "cuda_runtime_api.h")):
        pytest.skip("needs g++ and the CUDA headers")
    src, exe = tmp_path / "per_device.cpp", tmp_path / "per_device"
    src.write_text(PROGRAM)
    subprocess.run([gxx, "-std=c++17", "-O1", "-pthread", "-I", os.path.join(cuda, "include"),
                    "-I", CSRC, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout


def test_no_launcher_sets_a_limit_once_per_process():
    for path in glob.glob(os.path.join(CSRC, "*.cu*")):
        text = open(path).read()
        assert "call_once" not in text and "cudaFuncSetAttribute" not in text, path
