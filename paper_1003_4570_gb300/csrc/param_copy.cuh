// Small host tables to the device as the parameters of launches that write them.  Parameters are read
// when a launch is made, so the host array may go when the call returns, nothing waits, and a captured
// graph holds the values; a copy from pageable memory may be pending until the next synchronisation.
#pragma once

#include <cuda_runtime.h>

#include <algorithm>
#include <cstring>

struct ParamChunk {
  unsigned long long w[496];   // with the other parameters below 4 KB
};

static __global__ void __launch_bounds__(128) param_copy_kernel(const __grid_constant__ ParamChunk c, int n,
                                                                unsigned long long* __restrict__ dst) {
  for (int i = threadIdx.x; i < n; i += 128) dst[i] = c.w[i];
}

// `bytes` (a multiple of 8) from src to dst (8-byte aligned) on the stream.
inline cudaError_t copy_as_params(cudaStream_t st, void* dst, const void* src, size_t bytes) {
  for (size_t at = 0; at < bytes; at += sizeof(ParamChunk)) {
    ParamChunk c;
    const size_t n = std::min(sizeof(ParamChunk), bytes - at);
    std::memcpy(c.w, static_cast<const char*>(src) + at, n);
    param_copy_kernel<<<1, 128, 0, st>>>(c, (int)(n / 8), reinterpret_cast<unsigned long long*>(static_cast<char*>(dst) + at));
  }
  return cudaGetLastError();
}
