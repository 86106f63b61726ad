"""The last-block reduction on the host: its source is compiled as C++ with a thread per CUDA thread,
and every read of another block's value must follow a fence that the reading thread ran after its
block had counted the others (the acquire side of the counter pattern; a race otherwise)."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

HOST = r"""
#include <barrier>
#include <cmath>
#include <cstdio>
#include <thread>
#include <vector>
#include <cuda_runtime.h>
using std::fma;

constexpr int NT = 256;
struct Dim { unsigned x; };
static thread_local Dim threadIdx;
static Dim blockIdx, gridDim;
static thread_local int fences;       // fences of this thread since its block's count was seen
static bool counted;                  // this block has counted itself and the others
static int unordered = 0;
static std::barrier<> block_barrier(NT);
static std::vector<std::barrier<>*> warp_barrier;
static double lane[NT];

static void __syncthreads() { block_barrier.arrive_and_wait(); }
static void __threadfence() { if (counted) ++fences; }
static unsigned atomicAdd(unsigned* c, unsigned v) { unsigned o = *c; *c += v; counted = true; return o; }
static double __shfl_xor_sync(unsigned, double a, int o) {
  auto& b = *warp_barrier[threadIdx.x / 32];
  lane[threadIdx.x] = a;
  b.arrive_and_wait();
  const double r = lane[threadIdx.x ^ o];
  b.arrive_and_wait();
  return r;
}
static double __ldcg(const double* p) {
  if (fences == 0) __atomic_fetch_add(&unordered, 1, __ATOMIC_RELAXED);
  return *p;
}
#include "kernels.h"

int main() {
  for (int w = 0; w < NT / 32; ++w) warp_barrier.push_back(new std::barrier<>(32));
  int bad = 0;
  for (unsigned blocks : {1u, 3u, 260u}) {
    std::vector<double> partials(blocks);
    unsigned counter = 0;
    double got = 0;
    gridDim.x = blocks;
    for (unsigned b = 0; b < blocks; ++b) {
      blockIdx.x = b;
      counted = false;
      double red[8];
      bool last = false;
      std::vector<std::thread> ts;
      for (int t = 0; t < NT; ++t)
        ts.emplace_back([&, t] {
          threadIdx.x = (unsigned)t;
          fences = 0;
          double a = 1.0 + b;
          if (pcexp::grid_reduce<pcexp::SumOf>(a, red, last, partials.data(), &counter)) got = a;
        });
      for (auto& t : ts) t.join();
    }
    const double want = 256.0 * (blocks + blocks * (blocks - 1.0) / 2);
    if (got != want || counter != 0) ++bad;
  }
  std::printf("%d %d\n", bad, unordered);
  return 0;
}
"""


def test_reads_of_other_blocks_follow_a_fence(tmp_path):
    if shutil.which("g++") is None or not os.path.isdir("/usr/local/cuda/include"):
        pytest.skip("no host compiler or CUDA headers")
    src = tmp_path / "reduce.cpp"
    src.write_text(HOST)
    exe = str(tmp_path / "reduce")
    subprocess.run(["g++", "-std=c++20", "-O1", "-w", "-pthread", "-I/usr/local/cuda/include",
                    "-I", os.path.join(ROOT, "paper_1801_06300_gb300", "csrc"), str(src), "-o", exe], check=True)
    bad, unordered = map(int, subprocess.run([exe], check=True, capture_output=True, text=True, timeout=300).stdout.split())
    assert bad == 0, "wrong sum"
    assert unordered == 0, f"{unordered} reads of other blocks' values without a fence before them"
