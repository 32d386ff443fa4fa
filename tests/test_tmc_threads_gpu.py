"""Tensor-matrix contractions from several host threads at once: two shapes that
run the same kernel with different amounts of shared memory.  The threads are
C++ (Python's lock keeps calls from overlapping closely enough)."""
import os
import subprocess

import pytest

pytestmark = pytest.mark.gpu

tg = pytest.importorskip("paper_2501_03121_gb300")

SOURCE = r"""
#include <cuda_runtime.h>
#include <dlfcn.h>
#include <stdio.h>
#include <atomic>
#include <thread>
#include <vector>
#include "tvc.h"
int main(int, char** argv) {
  void* h = dlopen(argv[1], RTLD_NOW);
  auto call = (decltype(&::tmc))dlsym(h, "tmc");
  auto size = (decltype(&::tmc_workspace_size))dlsym(h, "tmc_workspace_size");
  const int64_t dims[2][3] = {{2, 256, 1200}, {1000, 32, 1}};
  const int64_t R = 16, entries[2] = {2 * 256 * 1200, 32000}, outputs[2] = {2 * 16 * 1200, 16 * 32};
  std::atomic<int> failed{0};
  std::vector<std::thread> threads;
  for (int t = 0; t < 4; t++)
    threads.emplace_back([&, t] {
      const int c = t & 1, order = 3 - c, mode = 1 - c;
      const size_t need = size(order, dims[c], mode, R, TVC_F32);
      float *A, *X, *Y;
      void* w;
      cudaStream_t s;
      bool ok = cudaSetDevice(0) == cudaSuccess && cudaMalloc(&A, entries[c] * 4) == cudaSuccess &&
                cudaMalloc(&X, R * 1000 * 4) == cudaSuccess && cudaMalloc(&Y, outputs[c] * 4) == cudaSuccess &&
                cudaMalloc(&w, need + 1) == cudaSuccess &&
                cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking) == cudaSuccess;
      ok = ok && cudaMemset(A, 0, entries[c] * 4) == cudaSuccess && cudaMemset(X, 0, R * 1000 * 4) == cudaSuccess &&
           cudaDeviceSynchronize() == cudaSuccess;
      for (int i = 0; ok && i < 20000; i++)
        if (call(A, order, dims[c], mode, X, R, Y, TVC_F32, nullptr, 1.0, 0.0, w, need, s) != TVC_OK) failed++;
      if (!ok || cudaStreamSynchronize(s) != cudaSuccess) failed++;
    });
  for (auto& t : threads) t.join();
  printf("failed %d\n", failed.load());
}
"""


def test_two_shapes_of_one_kernel(tmp_path):
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    src, exe = tmp_path / "threads.cpp", tmp_path / "threads"
    src.write_text(SOURCE)
    subprocess.run(["nvcc", "-O2", "-std=c++17", "-I", os.path.join(root, "include"), str(src), "-o", str(exe), "-ldl"],
                   check=True)
    lib = os.path.join(root, "paper_2501_03121_gb300", "_lib", "libtvc_gb300.so")
    out = subprocess.run([str(exe), lib], capture_output=True, text=True, timeout=300)
    assert out.stdout.strip() == "failed 0", out.stdout + out.stderr
