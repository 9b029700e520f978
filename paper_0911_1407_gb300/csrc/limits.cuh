// limits.cuh -- dynamic shared-memory limits of the kernels.
#pragma once

#include <atomic>

#include "ctx.h"

namespace plc {

inline int current_device() {
  int dev = 0;
  check(cudaGetDevice(&dev), "cudaGetDevice");
  return dev;
}

// Raise a kernel's dynamic shared-memory limit (also below 48 KB, which is the
// limit for its static and dynamic shared memory together), once for the
// kernel and the current device dev: the attribute belongs to the device's copy of
// the function, and contexts of one process may live on several devices.
// Devices beyond the 64th are set on every call.  Setting it twice (two threads
// at their first launch) does no harm.
template <auto Kernel> inline void set_smem4(int dev, size_t bytes) {
  constexpr int kMaxDevices = 64;
  static std::atomic<bool> set[kMaxDevices] = {};
  if (dev < kMaxDevices && set[dev].load(std::memory_order_acquire)) return;
  check(cudaFuncSetAttribute(Kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes),
        "cudaFuncSetAttribute");
  if (dev < kMaxDevices) set[dev].store(true, std::memory_order_release);
}

}  // namespace plc
