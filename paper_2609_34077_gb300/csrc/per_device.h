// Host values that belong to a device, found on each device's first use. Function-local statics would keep
// the first device's for all of them; a launch attribute set on one device does not hold on another.
// Not part of the C ABI.
#pragma once

#include <cuda_runtime.h>

#include <atomic>

namespace mcft {

constexpr int kMaxDevices = 64;

inline int current_device() {
  int dev = 0;
  cudaGetDevice(&dev);
  return dev;
}

// A positive number per device. make() may run more than once where threads meet on the first use (it
// gives the same number); what it gives is kept only if it is positive.
struct PerDeviceInt {
  std::atomic<int> value[kMaxDevices] = {};
  template <typename F>
  int get(F make) {
    const int dev = current_device();
    const bool known = dev >= 0 && dev < kMaxDevices;
    int v = known ? value[dev].load(std::memory_order_relaxed) : 0;
    if (v > 0) return v;
    v = make();
    if (known && v > 0) value[dev].store(v, std::memory_order_relaxed);
    return v;
  }
};

// A kernel's opt-in to more than 48 KB of dynamic shared memory, once per device. A failure is not kept.
struct SmemOptIn {
  PerDeviceInt done;
  cudaError_t allow(const void* kernel, int bytes) {
    cudaError_t e = cudaSuccess;
    done.get([&] {
      e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
      return e == cudaSuccess ? 1 : 0;
    });
    return e;
  }
};

// Clusters of a kernel that fit the device at once (0: none, or the query failed), found once per device.
struct ResidentClusters {
  PerDeviceInt clusters;
  int get(const void* kernel, int grid, int block, size_t smem) {
    return clusters.get([&] {
      cudaLaunchConfig_t cfg = {};
      cfg.gridDim = dim3(unsigned(grid));
      cfg.blockDim = dim3(unsigned(block));
      cfg.dynamicSmemBytes = smem;
      int n = 0;
      if (cudaOccupancyMaxActiveClusters(&n, kernel, &cfg) != cudaSuccess) {
        (void)cudaGetLastError();
        n = 0;
      }
      return n;
    });
  }
};

}  // namespace mcft
