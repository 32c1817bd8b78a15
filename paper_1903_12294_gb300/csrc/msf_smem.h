// Opting kernels into more than 48 KB of dynamic shared memory (host code only).
#pragma once

#include <cuda_runtime_api.h>
#include <stddef.h>
#include <stdint.h>

#include <atomic>

namespace msf {

// Allow `kernel` to be launched with `bytes` of dynamic shared memory on the current device. The
// attribute belongs to the function on one device, so `done` (one per kernel) has a bit per device.
// `bytes` is the most that any launch of the kernel asks for, the same at every call: contexts of
// several host threads then set nothing but this value, in any order. A repeated call costs one
// atomic load.
template <typename K>
inline void ensure_smem_attr(K kernel, size_t bytes, std::atomic<uint64_t>& done) {
  int dev = 0;
  cudaGetDevice(&dev);
  const uint64_t bit = dev >= 0 && dev < 64 ? 1ull << dev : 0ull;  // (beyond: set each time)
  if (done.load(std::memory_order_acquire) & bit) return;
  if (cudaFuncSetAttribute(reinterpret_cast<const void*>(kernel),
                           cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)bytes) == cudaSuccess)
    done.fetch_or(bit, std::memory_order_release);
}

}  // namespace msf
