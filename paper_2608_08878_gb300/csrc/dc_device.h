// dc_device.h -- what the library tells a device or asks of it once: kernel
// attributes and occupancy belong to one device, and handles on several devices
// may launch from several threads of a process.
#pragma once

#include <cuda_runtime.h>

#include <atomic>
#include <mutex>

namespace dc {

constexpr int kDevices = 64;  // ordinals whose answers are kept; others are told and asked on each call

// The current device's ordinal if its answers are kept, else -1.
inline int device_slot() {
  int dev = -1;
  return cudaGetDevice(&dev) == cudaSuccess && dev >= 0 && dev < kDevices ? dev : -1;
}

// One kernel's dynamic shared memory limit, raised once per device (a launcher's
// static). Threads that meet here set the same value twice.
class SmemLimit {
 public:
  template <class Kernel>
  cudaError_t raise(Kernel* kernel, int bytes) {
    const int dev = device_slot();
    if (dev >= 0 && done_[dev].load(std::memory_order_acquire)) return cudaSuccess;
    const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    if (e == cudaSuccess && dev >= 0) done_[dev].store(true, std::memory_order_release);
    return e;
  }

 private:
  std::atomic<bool> done_[kDevices] = {};
};

// A value that `ask` returns for the current device, asked once per device.
template <class T>
class PerDevice {
 public:
  template <class Ask>
  T get(Ask ask) {
    const int dev = device_slot();
    if (dev < 0) return ask();
    std::call_once(once_[dev], [&] { kept_[dev] = ask(); });
    return kept_[dev];
  }

 private:
  std::once_flag once_[kDevices];
  T kept_[kDevices] = {};
};

}  // namespace dc
