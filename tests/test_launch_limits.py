"""The dynamic shared-memory limit of a kernel (csrc/launch.cuh) with a stand-in for cudaFuncSetAttribute: a
host program, no GPU.  A launch must find its own need, whatever other threads have set in between."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROGRAM = r'''
#include <cuda_runtime.h>
#include <stdio.h>
#include <atomic>
#include <thread>
static std::atomic<int> limit_a{0}, limit_b{0}, refuse_above{1 << 30};
__global__ void ka(int) {}
__global__ void kb(float) {}
template <typename T> cudaError_t fake_set(T* f, cudaFuncAttribute, int v) {
  if (v > refuse_above) return cudaErrorInvalidValue;
  ((const void*)f == (const void*)ka ? limit_a : limit_b) = v;
  return cudaSuccess;
}
static cudaError_t fake_device(int* d) { *d = 0; return cudaSuccess; }
#define cudaFuncSetAttribute fake_set
#define cudaGetDevice fake_device
#include "launch.cuh"
using namespace mmp;
int main() {
  int bad = 0;
  bad += set_smem(ka, 48 * 1024) != cudaSuccess || limit_a != 0;            // within the default
  bad += 2 * (set_smem(ka, 100000) != cudaSuccess || limit_a < 100000);
  bad += 4 * (set_smem(ka, 60000) != cudaSuccess || limit_a < 100000);      // a smaller need does not lower it
  bad += 8 * (set_smem(kb, 70000) != cudaSuccess || limit_b != 70000);      // kernels apart
  refuse_above = 200000;
  bad += 16 * (set_smem(kb, 300000) == cudaSuccess || set_smem(kb, 80000) != cudaSuccess || limit_b < 80000);
  std::atomic<int> low{0};
  auto user = [&](size_t need) {
    for (int i = 0; i < 20000; ++i) { set_smem(ka, need); low += limit_a < (int)need; }
  };
  std::thread t(user, 150000), u(user, 90000);
  t.join();
  u.join();
  bad += 32 * (low != 0);
  printf("bad %d\n", bad);
  return bad;
}
'''


def test_limit_of_a_kernel_only_grows(tmp_path):
    from paper_2411_18194_gb300 import build
    src, exe = tmp_path / "limits.cu", tmp_path / "limits"
    src.write_text(PROGRAM)
    cmd = [build.nvcc(), "-std=c++17", "-I" + build.SRC, "-I" + os.path.join(ROOT, "include")] + build.ARCH + [
        "-o", str(exe), str(src)]
    r = subprocess.run(cmd, capture_output=True, text=True, timeout=600)
    assert r.returncode == 0, r.stdout + r.stderr
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stdout + r.stderr
