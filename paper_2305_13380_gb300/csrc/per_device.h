// per_device.h -- what a launcher finds out once per device.
#pragma once
#include <cuda_runtime.h>

#include <atomic>

namespace sphh {

// kValues numbers of the current device (resident blocks per SM, ...), found by
// find(v) at the first call on that device.  Function attributes and occupancy
// belong to a device, and a process may use several, each from threads of its
// own: threads that meet in a first call find the same values, and a find that
// fails is tried again at the next call.
template <int kValues>
class PerDevice {
 public:
  template <class Find>
  cudaError_t get(int (&v)[kValues], Find find) {
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const bool kept = dev >= 0 && dev < kMaxDevices;
    if (kept && known_[dev].load(std::memory_order_acquire)) {
      for (int i = 0; i < kValues; ++i) v[i] = value_[dev][i].load(std::memory_order_relaxed);
      return cudaSuccess;
    }
    e = find(v);
    if (e == cudaSuccess && kept) {
      for (int i = 0; i < kValues; ++i) value_[dev][i].store(v[i], std::memory_order_relaxed);
      known_[dev].store(true, std::memory_order_release);
    }
    return e;
  }

 private:
  static constexpr int kMaxDevices = 64;
  std::atomic<bool> known_[kMaxDevices] = {};
  std::atomic<int> value_[kMaxDevices][kValues] = {};
};

// Lets `kernel` be launched with `bytes` of dynamic shared memory on the current
// device, and the blocks of `threads` threads that an SM then holds (at least 1).
template <class Kernel>
cudaError_t opt_in(Kernel kernel, size_t bytes) {
  return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
}
template <class Kernel>
cudaError_t resident_blocks(Kernel kernel, int threads, size_t bytes, int* blocks) {
  const cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks, kernel, threads, bytes);
  if (*blocks < 1) *blocks = 1;
  return e;
}

}  // namespace sphh
