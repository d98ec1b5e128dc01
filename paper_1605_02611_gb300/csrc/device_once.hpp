// Set-up that the CUDA runtime keeps per device.
#pragma once
#include <atomic>
#include <cstdint>

namespace gbdmrg {

// true once f() has returned true on device dev (remembered for the first 64 devices of the process;
// safe from several threads, which may call f twice)
class DeviceOnce {
  std::atomic<uint64_t> done_{0};

 public:
  template <class F>
  bool operator()(int dev, F&& f) {
    const uint64_t bit = dev >= 0 && dev < 64 ? 1ULL << dev : 0;
    if (done_.load(std::memory_order_acquire) & bit) return true;
    if (!f()) return false;
    done_.fetch_or(bit, std::memory_order_release);
    return true;
  }
};

#ifdef __CUDACC__
// raises the kernel's limit of dynamic shared memory on the current device
template <class K>
bool allow_shared_memory(DeviceOnce& once, K* kernel, int bytes) {
  int dev = 0;
  return cudaGetDevice(&dev) == cudaSuccess && once(dev, [&] {
           return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes) == cudaSuccess;
         });
}
#endif

}  // namespace gbdmrg
