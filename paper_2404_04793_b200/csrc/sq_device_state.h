// What the launchers remember from one launch to the next, by device: a process may use several, and a kernel's
// attributes (its limit of dynamic shared memory, clusters above the portable size) belong to the device that was
// current when they were set.  Safe with several host threads: the worst is that two of them set up the same thing.
#pragma once
#include <cuda_runtime_api.h>

#include <atomic>

namespace sq {

constexpr int kMaxDevices = 64;  // (on a device beyond, nothing is remembered)

// A set-up that is done once on every device.  For static storage.
class PerDevice {
 public:
  template <class F>
  cudaError_t once(F set_up) {
    int dev = -1;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    const bool known = dev >= 0 && dev < kMaxDevices;
    if (known && done_[dev].load(std::memory_order_acquire)) return cudaSuccess;
    e = set_up();
    if (e == cudaSuccess && known) done_[dev].store(true, std::memory_order_release);
    return e;
  }

 private:
  std::atomic<bool> done_[kMaxDevices] = {};
};

// Allows `bytes` of dynamic shared memory to each of the kernels.
template <class... K>
inline cudaError_t allow_smem(PerDevice& state, size_t bytes, K... kern) {
  return state.once([&] {
    cudaError_t e = cudaSuccess;
    auto set = [&](auto k) {
      if (e == cudaSuccess) e = cudaFuncSetAttribute(reinterpret_cast<const void*>(k), cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
    };
    (set(kern), ...);
    return e;
  });
}

// SMs of the current device.
inline int sm_count() {
  static std::atomic<int> count[kMaxDevices] = {};
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess) return 148;  // (the launch that follows reports it)
  const bool known = dev >= 0 && dev < kMaxDevices;
  int n = known ? count[dev].load(std::memory_order_relaxed) : 0;
  if (n == 0) {
    if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 148;
    if (known) count[dev].store(n, std::memory_order_relaxed);
  }
  return n;
}

}  // namespace sq
