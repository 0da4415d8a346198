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

// Clusters of `ctas` CTAs of a kernel that the current device runs at a time, by size (up to 16).  For static
// storage, one per kernel and amount of shared memory; asked once for every size on every device.
class ClusterCount {
 public:
  int active(const void* kern, int ctas, int threads, size_t smem) {
    int dev = -1;
    if (ctas < 1 || ctas > kSizes || cudaGetDevice(&dev) != cudaSuccess) return 0;
    const bool known = dev >= 0 && dev < kMaxDevices;
    const int seen = known ? count_[dev][ctas - 1].load(std::memory_order_relaxed) : 0;
    if (seen) return seen - 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(ctas);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = ctas;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int n = 0;
    if (cudaOccupancyMaxActiveClusters(&n, kern, &cfg) != cudaSuccess) {
      cudaGetLastError();
      n = 0;
    }
    if (known) count_[dev][ctas - 1].store(n + 1, std::memory_order_relaxed);
    return n;
  }

 private:
  static constexpr int kSizes = 16;
  std::atomic<int> count_[kMaxDevices][kSizes] = {};
};

// Whether the current device holds a cluster of `ctas` CTAs of a kernel (which is allowed that size) with `smem` bytes
// of dynamic shared memory each.  Above the portable 8 that depends on the device and on what is left of it
// (partitions, disabled SMs).  For static storage, one per kernel; asked once for every size on every device, with the most smem
// that the kernel is launched with.
class ClusterFit {
 public:
  bool fits(const void* kern, int ctas, int threads, size_t smem) { return count_.active(kern, ctas, threads, smem) > 0; }

 private:
  ClusterCount count_;
};

// The most CTAs per cluster, up to `limit` and at least two, with room for `units` clusters at a time; 0 where there is none.
// room(ctas): how many clusters of that size the device runs at a time.
template <class Room>
inline int most_ctas(int limit, long long units, Room room) {
  while (limit >= 2 && room(limit) < units) --limit;
  return limit >= 2 ? limit : 0;
}

// launch(limit) with clusters of at most `limit` CTAs, and where the device does not hold those (or the plan does not
// work out) with at most the portable 8.
template <class F>
inline cudaError_t with_portable_clusters(int limit, F launch) {
  const cudaError_t e = launch(limit);
  return e == cudaErrorNotSupported && limit > 8 ? launch(8) : e;
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
