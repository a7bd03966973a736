// What a launch needs to know of its kernel on the current device. The opt-in to more than 48 KB of dynamic shared memory
// belongs to a device, so it is made once per kernel and device (one process may hold contexts on several).
#pragma once

#include <cuda_runtime.h>

#include <map>
#include <mutex>
#include <utility>

namespace fs {

struct LaunchSetup {
  cudaError_t err = cudaSuccess;
  int nsm = 0;
  int blocks_per_sm = 0;  // resident blocks of `threads` with `smem`
};

// smem: the largest dynamic shared memory `kern` is launched with. Any thread may call it; a failure is not kept.
inline LaunchSetup launch_setup(const void* kern, size_t smem, int threads) {
  static std::mutex m;
  static std::map<std::pair<int, const void*>, LaunchSetup> made;
  LaunchSetup s;
  int dev = 0;
  if ((s.err = cudaGetDevice(&dev))) return s;
  std::lock_guard<std::mutex> lock(m);
  auto it = made.find({dev, kern});
  if (it != made.end()) return it->second;
  s.err = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (!s.err) s.err = cudaDeviceGetAttribute(&s.nsm, cudaDevAttrMultiProcessorCount, dev);
  if (!s.err) s.err = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&s.blocks_per_sm, kern, threads, smem);
  if (!s.err && s.blocks_per_sm < 1) s.err = cudaErrorInvalidConfiguration;
  if (!s.err) made[{dev, kern}] = s;
  return s;
}

}  // namespace fs
