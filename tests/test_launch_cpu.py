"""The launch helpers of pp_launch.cuh against a stand-in for the CUDA runtime
(host compiler only): two host threads whose plans ask for different amounts
of shared memory of one kernel."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2005_11806_gb300", "csrc")

# What pp_launch.cuh uses of the runtime.  The function's limit is `limit`;
# `in_occupancy` is called while a thread asks for the occupancy.
FAKE = r"""
#pragma once
#include <cstddef>
#include <functional>
enum cudaError_t { cudaSuccess = 0, cudaErrorInvalidValue = 1 };
enum cudaFuncAttribute { cudaFuncAttributeMaxDynamicSharedMemorySize = 8 };
enum cudaDeviceAttr { cudaDevAttrMultiProcessorCount = 16, cudaDevAttrMaxSharedMemoryPerBlockOptin = 97 };
struct cudaFuncAttributes { size_t sharedSizeBytes; };
typedef struct Stream_* cudaStream_t;
typedef struct Graph_* cudaGraph_t;
typedef struct Node_* cudaGraphNode_t;
struct dim3 { unsigned x, y, z; dim3(unsigned a = 1, unsigned b = 1, unsigned c = 1) : x(a), y(b), z(c) {} };
struct cudaKernelNodeParams {
  void* func; dim3 gridDim, blockDim; unsigned sharedMemBytes; void** kernelParams; void** extra;
};
extern int limit, most, fixed_bytes;
extern std::function<void(size_t)> in_occupancy;
inline cudaError_t cudaGetLastError() { return cudaSuccess; }
inline cudaError_t cudaGetDevice(int* d) { *d = 0; return cudaSuccess; }
inline cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr a, int) {
  *v = a == cudaDevAttrMultiProcessorCount ? 152 : most;
  return cudaSuccess;
}
template <class F> cudaError_t cudaFuncGetAttributes(cudaFuncAttributes* a, F) {
  a->sharedSizeBytes = (size_t)fixed_bytes;
  return cudaSuccess;
}
template <class F> cudaError_t cudaFuncSetAttribute(F, cudaFuncAttribute, int v) {
  if (v + fixed_bytes > most) return cudaErrorInvalidValue;
  limit = v;
  return cudaSuccess;
}
template <class F> cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessor(int* n, F, int, size_t smem) {
  in_occupancy(smem);
  *n = 2;
  return cudaSuccess;
}
inline cudaError_t cudaLaunchKernel(const void*, dim3, dim3, void**, size_t, cudaStream_t) { return cudaSuccess; }
inline cudaError_t cudaGraphAddKernelNode(cudaGraphNode_t*, cudaGraph_t, const cudaGraphNode_t*, size_t,
                                          const cudaKernelNodeParams*) { return cudaSuccess; }
"""

MAIN = r"""
#include "pp_launch.cuh"
#include <cstdio>
#include <thread>
int limit = 48 * 1024, most = 232448, fixed_bytes = 512;
std::function<void(size_t)> in_occupancy = [](size_t) {};
void kernel(int) {}
int main() {
  const size_t large = 96000, small = 76800;  // the y kernel of FP64 plans with ny = 250 and ny = 200
  long long n = 0;
  bool once = false;
  // while the first thread is between its two calls, another one asks for less
  in_occupancy = [&](size_t smem) {
    if (smem == large && !once) {
      once = true;
      std::thread([&] { long long m = 0; pp::resident_blocks<&kernel>(256, small, &m); }).join();
    }
  };
  if (pp::resident_blocks<&kernel>(256, large, &n) != cudaSuccess || n != 304) return 1;
  std::printf("%d\n", limit >= (int)large);
  // the next launch of the same plan
  if (pp::resident_blocks<&kernel>(256, large, &n) != cudaSuccess || n != 304) return 1;
  std::printf("%d\n", limit >= (int)large);
  if (pp::resident_blocks<&kernel>(256, small, &n) != cudaSuccess) return 1;
  std::printf("%d\n", limit >= (int)large);
  std::printf("%d\n", limit + fixed_bytes <= most);
  return 0;
}
"""


def test_shared_memory_limit_is_never_lowered(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no host compiler")
    (tmp_path / "cuda_runtime.h").write_text(FAKE)
    (tmp_path / "main.cpp").write_text('#include <cstdint>\n#include "cuda_runtime.h"\n' + MAIN)
    exe = str(tmp_path / "main")
    r = subprocess.run([gxx, "-std=c++17", "-O1", "-pthread", "-I", str(tmp_path), "-I", CSRC,
                        str(tmp_path / "main.cpp"), "-o", exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    r = subprocess.run([exe], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0
    assert r.stdout.split() == ["1"] * 4
