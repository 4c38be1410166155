// Opt-in shared memory of a kernel.  The limit belongs to the kernel and the device, not to a launch, and several handles launch from
// several threads: it is only ever raised, one thread at a time, so that a launch never meets a limit that another one lowered.
#pragma once
#include <cuda_runtime.h>

#include <map>
#include <mutex>
#include <utility>

namespace amp {

inline cudaError_t allow_dynamic_smem(const void* kernel, const size_t bytes) {
  static std::mutex lock;
  static std::map<std::pair<const void*, int>, size_t> allowed;
  int device = 0;
  cudaError_t e = cudaGetDevice(&device);
  if (e != cudaSuccess) return e;
  std::lock_guard<std::mutex> hold(lock);
  size_t& most = allowed[{kernel, device}];
  if (bytes <= most) return cudaSuccess;
  e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
  if (e == cudaSuccess) most = bytes;
  return e;
}

}  // namespace amp
