// What the host asks a device for once: a kernel's resident blocks, its cluster
// size, its shared-memory opt-in.  Kernel attributes belong to the device that is
// current when they are set, so a process that works on a second device asks and
// sets again there.
#pragma once
#include <atomic>

#include <cuda_runtime.h>

namespace ps {

// A positive int per device, from query(&value) at the first use on each (several
// threads may ask at once: they store the same answer).
class PerDevice {
 public:
  template <typename F>
  cudaError_t get(F query, int* out) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const bool kept = dev >= 0 && dev < kDevices;
    int v = kept ? v_[dev].load(std::memory_order_relaxed) : 0;
    if (v == 0) {
      if ((e = query(&v)) != cudaSuccess) return e;
      if (v < 1) v = 1;
      if (kept) v_[dev].store(v, std::memory_order_relaxed);
    }
    *out = v;
    return cudaSuccess;
  }

 private:
  static constexpr int kDevices = 64;
  std::atomic<int> v_[kDevices] = {};
};

// Resident blocks of a kernel per SM with `smem` bytes of dynamic shared memory,
// which it is opted in for at the first use on a device.
template <typename K>
inline cudaError_t resident_blocks(K kern, int threads, int smem, PerDevice& cache, int* out) {
  return cache.get(
      [&](int* n) {
        const void* k = (const void*)kern;
        const cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        return e != cudaSuccess ? e : cudaOccupancyMaxActiveBlocksPerMultiprocessor(n, k, threads, smem);
      },
      out);
}

}  // namespace ps
