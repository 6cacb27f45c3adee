"""The barrier of the one-launch power iteration (power.cuh), in a kernel of its own: blocks
see what the others wrote before it, also while the arrival count passes 2^32, and a wait
for a block that never arrives gives up after its limit, sets the error word and lets the
kernel end."""
import subprocess

import pytest

from paper_2412_09734_gb300.build import ARCH, CSRC, nvcc

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include <chrono>
#include <cstdio>
#include "power.cuh"
using namespace mpax;

// Blocks from `present` on never arrive.  Round r: every block writes its cell, meets the
// others and reads the next one's cell, which holds r or, when that block is ahead, r + 1.
__global__ void meet(GridBar b, unsigned start, int rounds, int present, unsigned long long limit,
                     volatile int* cell, int* wrong, int* gave_up) {
  if ((int)blockIdx.x >= present) return;
  unsigned phase = start;
  for (int r = 1; r <= rounds; ++r) {
    if (threadIdx.x == 0) cell[blockIdx.x] = r;
    if (!grid_sync(b, phase, limit)) {
      if (threadIdx.x == 0) gave_up[blockIdx.x] = 1;
      return;
    }
    if (threadIdx.x == 31) {
      const int v = cell[(blockIdx.x + 1) % gridDim.x];
      if (v != r && v != r + 1) atomicAdd(wrong, 1);
    }
  }
}

int main() {
  constexpr int kBlocks = 16;
  unsigned* w;
  int* out;  // cells, wrong, gave_up
  cudaMalloc(&w, sizeof(unsigned) * kGridBarWords);
  cudaMalloc(&out, sizeof(int) * (2 * kBlocks + 1));
  const unsigned starts[3] = {0u, 0u - 40u * kBlocks, 0u};
  for (int t = 0; t < 3; ++t) {
    const int present = t < 2 ? kBlocks : kBlocks - 1, rounds = t < 2 ? 100 : 1;
    const unsigned long long limit = t < 2 ? kWaitNs : 20000000ull;  // 20 ms
    unsigned words[kGridBarWords] = {starts[t], 0u, 0u};
    cudaMemcpy(w, words, sizeof(words), cudaMemcpyHostToDevice);
    cudaMemset(out, 0, sizeof(int) * (2 * kBlocks + 1));
    const auto t0 = std::chrono::steady_clock::now();
    cudaError_t e = launch_cooperative(meet, kBlocks, 64, 0, (cudaStream_t)0, GridBar{w}, starts[t],
                                       rounds, present, limit, (volatile int*)out, out + kBlocks,
                                       out + kBlocks + 1);
    if (!e) e = cudaDeviceSynchronize();
    const double ms = std::chrono::duration<double, std::milli>(
        std::chrono::steady_clock::now() - t0).count();
    int h[2 * kBlocks + 1];
    cudaMemcpy(h, out, sizeof(h), cudaMemcpyDeviceToHost);
    cudaMemcpy(words, w, sizeof(words), cudaMemcpyDeviceToHost);
    int up = 0;
    for (int b = 0; b < kBlocks; ++b) up += h[kBlocks + 1 + b];
    std::printf("%d %d %d %u %u %f\n", (int)e, h[kBlocks], up, words[0] - starts[t], words[2], ms);
  }
}
"""


def test_barrier_meets_wraps_and_gives_up(tmp_path):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    src, exe = tmp_path / "barrier.cu", tmp_path / "barrier"
    src.write_text(SOURCE)
    subprocess.run([nvcc(), *ARCH, "-O3", "-std=c++17", "-I", CSRC, "-o", str(exe), str(src)],
                   check=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True, timeout=60).stdout
    plain, wrap, missing = ([float(v) for v in line.split()] for line in out.splitlines())
    for err, wrong, up, arrived, flag, _ in (plain, wrap):
        assert (err, wrong, up, arrived, flag) == (0, 0, 0, 1600, 0)
    err, _, up, arrived, flag, ms = missing
    assert (err, up, arrived, flag) == (0, 15, 15, 1)
    assert 20.0 <= ms < 1000.0
