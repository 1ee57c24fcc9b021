// Host helpers for per-device launch state: raise a kernel's dynamic
// shared-memory limit to at least a launch's need, never lowering it, and the
// device's SM count.  Handles of different geometries, devices and host
// threads share one kernel instantiation.  A limit belongs to the device that
// is current when it is set, so it is recorded per device; on each the limit a
// launch sees must be the largest any launch asked for, and the check and the
// update run under one process-wide lock.
#pragma once

#include <cuda_runtime.h>

#include <atomic>
#include <cstddef>
#include <mutex>

namespace mra {

constexpr int kDeviceRecords = 64;  // devices with a higher number set the limit and ask for the count each time

inline std::mutex &smem_limit_mutex() {
  static std::mutex m;
  return m;
}

// A kernel's record of the limits already set, per device.
struct SmemLimit {
  size_t granted[kDeviceRecords] = {};
};

template <class Kernel>
cudaError_t raise_smem_limit(Kernel *kernel, size_t bytes, SmemLimit &limit) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  std::lock_guard<std::mutex> lock(smem_limit_mutex());
  if (dev < kDeviceRecords && limit.granted[dev] >= bytes) return cudaSuccess;
  e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(bytes));
  if (e == cudaSuccess && dev < kDeviceRecords) limit.granted[dev] = bytes;
  return e;
}

// SMs of the current device.
inline cudaError_t sm_count(int *sms) {
  static std::atomic<int> count[kDeviceRecords];
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  *sms = dev < kDeviceRecords ? count[dev].load(std::memory_order_relaxed) : 0;
  if (*sms > 0) return cudaSuccess;
  e = cudaDeviceGetAttribute(sms, cudaDevAttrMultiProcessorCount, dev);
  if (e == cudaSuccess && dev < kDeviceRecords) count[dev].store(*sms, std::memory_order_relaxed);
  return e;
}

}  // namespace mra
