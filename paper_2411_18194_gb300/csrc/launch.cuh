// launch.cuh -- small host helpers shared by the launchers.
#pragma once
#include <algorithm>
#include <map>
#include <mutex>
#include <utility>

#include "kernels.h"

namespace mmp {

static inline int grid_for(long long n, int threads) {
  long long b = (n + threads - 1) / threads;
  return (int)(b > 152 * 16 ? 152 * 16 : (b < 1 ? 1 : b));
}

inline cudaError_t raise_smem_limit(const void* kernel, size_t bytes) {
  static std::mutex mu;
  static std::map<std::pair<const void*, int>, size_t> limits;   // by kernel and device
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  std::lock_guard<std::mutex> lk(mu);
  size_t& limit = limits[{kernel, dev}];
  const size_t want = std::max(limit, bytes);
  e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)want);
  if (e == cudaSuccess) limit = want;
  return e;
}

// Dynamic shared memory above the default limit (fixed: the kernel's static shared
// memory).  The limit belongs to the kernel, not to the launch: it only grows, or a
// context on another host thread with a smaller need could lower it between this
// call and the launch.
template <typename K>
static inline cudaError_t set_smem(K kernel, size_t bytes, size_t fixed = 0) {
  if (bytes + fixed <= 48 * 1024) return cudaSuccess;
  return raise_smem_limit(reinterpret_cast<const void*>(kernel), bytes);
}

// A kernel that may be placed while its predecessor in the stream drains: its
// blocks wait in after_predecessor() until that grid is complete and its
// writes are visible.  Every kernel launched this way calls it in every thread
// before its first access to memory that an earlier launch writes or reads, so
// the grids of a chain still complete in order.  `chain` false: a plain launch.
// In a stream this takes the launch latency off each pass (demag field of
// 128x100x4, three launches: 26.6 -> 22.2 us); between the nodes of a graph it
// costs more than it gives (64x64x1, ten fixed steps: 1051 -> 1160 us), so graphs
// are captured without it.
template <typename... P, typename... A>
static inline cudaError_t launch_chained(bool chain, void (*kernel)(P...), dim3 grid, int threads, size_t smem,
                                         cudaStream_t s, const A&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = chain ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kernel, args...);
}

// (no effect in a kernel launched without the attribute)
__device__ __forceinline__ void after_predecessor() {
  asm volatile("griddepcontrol.wait;\n" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");
}

}  // namespace mmp
