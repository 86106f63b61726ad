"""A kernel that needs a raised shared-memory limit has it on every device it is launched on: the
library's own launchers run here against a stand-in for the CUDA runtime with two devices."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

FAKE = r"""
#include <cstdio>
#include <cstring>
#include <map>
#include <utility>
#include <cmath>
#include <cuda_runtime.h>
using std::fma;
// names of device code in the header's templates, never called here
static struct { unsigned x; } threadIdx, blockIdx, gridDim;
void __syncthreads();
void __threadfence();
unsigned atomicAdd(unsigned*, unsigned);
double __shfl_xor_sync(unsigned, double, int);
double __ldcg(const double*);
#include "kernels.h"

static int device = 0, missing = 0, launches = 0;
static std::map<std::pair<const void*, int>, int> limit;  // (kernel, device) -> raised limit
static dim3 grid, block;
static size_t smem;
static void* stream;

static cudaError_t launch(const void* f, size_t bytes) {
  ++launches;
  // raised somewhere: needed everywhere
  for (auto& l : limit)
    if (l.first.first == f && (!limit.count({f, device}) || limit[{f, device}] < (int)bytes)) {
      ++missing;
      return cudaErrorInvalidValue;
    }
  return cudaSuccess;
}
extern "C" {
void** __cudaRegisterFatBinary(void*) { static void* h; return &h; }
void __cudaRegisterFatBinaryEnd(void**) {}
void __cudaUnregisterFatBinary(void**) {}
void __cudaRegisterFunction(void**, const char*, char*, const char*, int, uint3*, uint3*, dim3*, dim3*, int*) {}
unsigned __cudaPushCallConfiguration(dim3 g, dim3 b, size_t s, void* st) {
  grid = g; block = b; smem = s; stream = st;
  return 0;
}
cudaError_t __cudaPopCallConfiguration(dim3* g, dim3* b, size_t* s, void* st) {
  *g = grid; *b = block; *s = smem; *(void**)st = stream;
  return cudaSuccess;
}
cudaError_t __cudaGetKernel(cudaKernel_t* k, const void* f) { *k = (cudaKernel_t)f; return cudaSuccess; }
cudaError_t __cudaLaunchKernel(cudaKernel_t k, dim3, dim3, void**, size_t s, cudaStream_t) { return launch((const void*)k, s); }
cudaError_t cudaLaunchKernel(const void* f, dim3, dim3, void**, size_t s, cudaStream_t) { return launch(f, s); }
cudaError_t cudaLaunchKernelExC(const cudaLaunchConfig_t* c, const void* f, void**) { return launch(f, c->dynamicSmemBytes); }
cudaError_t cudaFuncSetAttribute(const void* f, cudaFuncAttribute a, int v) {
  if (a == cudaFuncAttributeMaxDynamicSharedMemorySize) limit[{f, device}] = v;
  return cudaSuccess;
}
cudaError_t cudaGetDevice(int* d) { *d = device; return cudaSuccess; }
cudaError_t cudaGetLastError(void) { return cudaSuccess; }
cudaError_t cudaDeviceGetAttribute(int* v, cudaDeviceAttr a, int) {
  *v = a == cudaDevAttrMultiProcessorCount ? 152 : 1;
  return cudaSuccess;
}
cudaError_t cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int* n, const void*, int, size_t, unsigned) {
  *n = 1;
  return cudaSuccess;
}
}

int main() {
  using namespace pcexp;
  KState* ks = nullptr;
  int bad = 0;
  for (int pass = 0; pass < 2; ++pass)
    for (device = 0; device < 2; ++device) {
      bad += launch_phi(ks, nullptr, 1.0, 1.0, nullptr, 0, nullptr, 1, nullptr) != cudaSuccess;
      bad += launch_phi_check(ks, nullptr, 1e-6, nullptr) != cudaSuccess;
      bad += launch_phi_adjoint(nullptr, 4, 4, 1.0, nullptr, nullptr, nullptr, nullptr) != cudaSuccess;
      const ColumnPlan p = plan_cgs_column<double>(1 << 16);  // a context plans on its own device
      unsigned long long slot = 0;
      bad += p.blocks < 1;
      bad += launch_cgs_column<double>(p, nullptr, 1 << 16, 1 << 16, 0, nullptr, nullptr, ks, &slot, 1e-12, false,
                                       nullptr) != cudaSuccess;
    }
  std::printf("%d %d %d\n", bad, missing, launches);
  return 0;
}
"""


def test_limits_are_raised_on_every_device(tmp_path):
    if shutil.which("nvcc") is None and not os.path.exists("/usr/local/cuda/bin/nvcc"):
        pytest.skip("no CUDA toolkit to build the library")
    from paper_1801_06300_gb300 import build
    build()
    pkg = os.path.join(ROOT, "paper_1801_06300_gb300")
    obj = os.path.join(pkg, "_build", "krylov_kernels.cu.o")
    if not os.path.exists(obj):
        pytest.skip("the library was built without its objects")
    src = tmp_path / "fake.cpp"
    src.write_text(FAKE)
    exe = str(tmp_path / "fake")
    subprocess.run(["g++", "-std=c++17", "-O1", "-w", "-I/usr/local/cuda/include", "-I", os.path.join(pkg, "csrc"),
                    str(src), obj, "-o", exe, "-lpthread"], check=True)
    bad, missing, launches = map(int, subprocess.run([exe], check=True, capture_output=True, text=True,
                                                     timeout=60).stdout.split())
    assert launches == 16
    assert missing == 0, f"{missing} launches on a device where the kernel's limit was not raised"
    assert bad == 0
