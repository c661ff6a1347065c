// Dynamic shared memory above 48 KB needs a kernel's limit raised first.  The limit belongs to the
// kernel, not to the caller: contexts of several host threads share it, so it is only ever raised.
// (Set to what each call needs, a small call would lower it between another thread's setting and its
// launch, which then fails.)  cudaFuncSetAttribute costs a driver call, made only when a launch needs
// more than the largest value already set.
#pragma once

#include <cuda_runtime.h>

#include <map>
#include <mutex>
#include <utility>

constexpr size_t kMaxDynamicSmem = 227 * 1024;   // a block's most on sm_103

template <typename K>
inline cudaError_t smem_limit(K kernel, size_t bytes) {
  static std::mutex mu;
  static std::map<std::pair<int, const void*>, size_t> current;   // per (device, kernel)
  if (bytes <= 48 * 1024) return cudaSuccess;
  int dev = 0;
  cudaGetDevice(&dev);
  std::lock_guard<std::mutex> lock(mu);
  size_t& cur = current[{dev, reinterpret_cast<const void*>(kernel)}];
  if (bytes <= cur) return cudaSuccess;
  const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
  if (e == cudaSuccess) cur = bytes;
  return e;
}
