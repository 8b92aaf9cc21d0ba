"""The host side of the convolutions, compiled with stand-ins for the CUDA runtime's calls and
run without a GPU (no kernel runs; the launches are recorded by the kernel whose shared-memory
limit the host raised before each)."""

import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1707_09898_gb300", "csrc")

HARNESS = r"""
#include <cuda.h>
#include <cuda_runtime.h>
#include <cstdio>
#include <cstring>
#include <map>
#include <set>
#include <string>
static int g_device = 0;
static bool g_maps = true;
static std::map<int, std::set<const void*>> g_raised;  // device -> kernels with a raised limit
static cudaError_t fake_get_device(int* d) { *d = g_device; return cudaSuccess; }
static cudaError_t fake_device_attribute(int* v, cudaDeviceAttr, int) { *v = 152; return cudaSuccess; }
template <typename K> static cudaError_t fake_set_attribute(K k, cudaFuncAttribute, int) {
  g_raised[g_device].insert(reinterpret_cast<const void*>(k));
  return cudaSuccess;
}
static CUresult fake_encode(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                            const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                            CUtensorMapL2promotion, CUtensorMapFloatOOBfill) {
  return g_maps ? CUDA_SUCCESS : CUDA_ERROR_INVALID_VALUE;
}
static cudaError_t fake_entry(const char*, void** f, unsigned, unsigned long long, cudaDriverEntryPointQueryResult* q) {
  *f = reinterpret_cast<void*>(&fake_encode);
  *q = cudaDriverEntryPointSuccess;
  return cudaSuccess;
}
static cudaError_t fake_peek() { return cudaSuccess; }
#define cudaGetDevice fake_get_device
#define cudaDeviceGetAttribute fake_device_attribute
#define cudaFuncSetAttribute fake_set_attribute
#define cudaGetDriverEntryPointByVersion fake_entry
#define cudaPeekAtLastError fake_peek
#include "unet.cu"

alignas(16) static char mem[64];
static int calls(int W, int r[3]) {  // 2 x 4 x 5 x W voxels, 32 -> 16 channels; no kernel runs, nothing is read
  float* f = reinterpret_cast<float*>(mem);
  r[0] = tmn_conv3d_forward(mem, mem, f, mem, 2, 4, 5, W, 32, 16, 1, nullptr);
  r[1] = tmn_conv3d_backward_data(f, mem, f, 2, 4, 5, W, 32, 16, 0, nullptr);
  r[2] = tmn_conv3d_backward_weight(mem, f, f, f, f, 1 << 22, 2, 4, 5, W, 32, 16, nullptr);
  return r[0] || r[1] || r[2];
}
int main(int argc, char** argv) {
  int r[3];
  const std::set<const void*> gather = {(const void*)k_conv_tc<0, 16>, (const void*)k_conv_tc<1, 32>,
                                        (const void*)k_conv_dw_tc<16>};
  if (!strcmp(argv[1], "no_maps")) {
    g_maps = false;
    for (int W : {16, 32, 64}) {
      calls(W, r);
      printf("%d %d %d %d\n", W, r[0], r[1], r[2]);
    }
    for (const void* k : gather) printf("gather %d\n", (int)g_raised[0].count(k));
  } else {  // the same calls on two devices raise the limits of the same kernels on each
    for (int W : {8, 12, 16, 32, 64})
      for (g_device = 0; g_device < 2; g_device++)
        if (calls(W, r)) printf("failed %d %d %d\n", r[0], r[1], r[2]);
    printf("same %d of %d\n", (int)(g_raised[0] == g_raised[1]), (int)g_raised[0].size());
  }
  return 0;
}
"""


@pytest.fixture(scope="module")
def harness(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("no nvcc")
    d = tmp_path_factory.mktemp("conv_host")
    src, exe = str(d / "harness.cu"), str(d / "harness")
    with open(src, "w") as f:
        f.write(HARNESS)
    subprocess.run([nvcc, "-gencode", "arch=compute_103a,code=compute_103a", "-O0", "-std=c++17", "-w", "-I", CSRC, "-I",
                    os.path.join(ROOT, "include"), "-o", exe, src], check=True, capture_output=True, text=True)
    return lambda mode: subprocess.run([exe, mode], check=True, capture_output=True, text=True, timeout=60).stdout.split("\n")


def test_without_tensor_maps_the_gather_kernels_run(harness):
    """Where no tensor map can be made, the calls take the kernels that need none."""
    out = harness("no_maps")
    assert out[:3] == ["16 0 0 0", "32 0 0 0", "64 0 0 0"], out
    assert out[3:6] == ["gather 1"] * 3, out
