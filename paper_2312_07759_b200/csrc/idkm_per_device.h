// What is set once per kernel AND device: a kernel's shared-memory limit belongs to the device that was current when it was
// raised, and one process may use several, from several threads.
#pragma once
#include <atomic>

namespace idkm {

class PerDevice {
  std::atomic<unsigned long long> done_{0};

 public:
  // Runs set() unless it has succeeded on device `dev` before; returns its status (zero: success).
  template <class Set>
  auto once(int dev, Set set) -> decltype(set()) {
    using Status = decltype(set());
    const unsigned long long bit = (dev >= 0 && dev < 64) ? 1ull << dev : 0ull;   // (beyond the 64th: set on every call)
    if (done_.load(std::memory_order_acquire) & bit) return Status(0);
    const Status rc = set();
    if (rc == Status(0)) done_.fetch_or(bit, std::memory_order_release);
    return rc;
  }
};

#ifdef __CUDACC__
// Lets `func` be launched with `bytes` of dynamic shared memory on the current device.
template <class Kernel>
inline cudaError_t allow_smem(PerDevice& per_device, Kernel func, int bytes) {
  int dev = -1;
  const cudaError_t rc = cudaGetDevice(&dev);
  if (rc != cudaSuccess) return rc;
  return per_device.once(dev, [&] { return cudaFuncSetAttribute(func, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes); });
}
#endif

}  // namespace idkm
