"""Settings that belong to one device are made on every device that launches, checked without a GPU
with stand-ins for the runtime's calls."""

import os
import shutil
import subprocess

import pytest

from test_conv_host import CSRC, harness  # noqa: F401

HARNESS = r"""
#include <cuda_runtime.h>
#include <cstdio>
static int g_device = 0, g_sets[100], g_bytes[100];
static bool g_fail = false;
static cudaError_t fake_get_device(int* d) { *d = g_device; return cudaSuccess; }
static cudaError_t fake_device_attribute(int* v, cudaDeviceAttr, int d) { *v = 100 + d; return cudaSuccess; }
template <typename K> static cudaError_t fake_set_attribute(K, cudaFuncAttribute, int v) {
  if (g_fail) return cudaErrorInvalidValue;
  g_sets[g_device]++;
  g_bytes[g_device] = v;
  return cudaSuccess;
}
#define cudaGetDevice fake_get_device
#define cudaDeviceGetAttribute fake_device_attribute
#define cudaFuncSetAttribute fake_set_attribute
#include "device.cuh"
__global__ void kernel_a() {}
__global__ void kernel_b() {}
int main() {
  auto at = [](int d, size_t bytes) {
    g_device = d;
    return (int)tmk::allow_smem<kernel_a>(bytes);
  };
  at(0, 60000), at(0, 60000), at(1, 60000), at(0, 50000), at(0, 70000), at(0, 60000), at(90, 60000), at(90, 60000);
  printf("%d %d %d %d %d\n", g_sets[0], g_sets[1], g_sets[90], g_bytes[0], g_bytes[1]);
  g_device = 1;
  tmk::allow_smem<kernel_b>(60000);
  printf("%d\n", g_sets[1]);
  g_fail = true;
  printf("%d ", at(2, 60000));
  g_fail = false;
  const int again = at(2, 60000);
  printf("%d %d\n", again, g_sets[2]);
  for (int d : {0, 1, 0, 90}) {
    g_device = d;
    printf("%d ", tmk::sm_count());
  }
  return 0;
}
"""


def test_limits_and_sm_counts_per_device(tmp_path):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("no nvcc")
    src, exe = str(tmp_path / "h.cu"), str(tmp_path / "h")
    with open(src, "w") as f:
        f.write(HARNESS)
    subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=compute_103a", "-std=c++17", "-I", CSRC, "-o", exe, src],
                   check=True, capture_output=True, text=True)
    out = subprocess.run([exe], check=True, capture_output=True, text=True, timeout=60).stdout.split("\n")
    # raised once for 60000 and once more for 70000 on device 0, once on device 1, every time past the table
    assert out[:4] == ["2 1 2 70000 60000", "2", "0 1 1", "100 101 100 190 "], out


def test_convolutions_on_a_second_device(harness):  # noqa: F811
    """Every kernel whose limit is raised for a call on one device has it raised on the other."""
    out = harness("devices")
    assert out[0].startswith("same 1 of "), out
    assert int(out[0].split()[-1]) >= 14, out  # forward, data and weight gradients of five row lengths
