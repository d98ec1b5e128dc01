// Which vectors of a caller the kernels may read or write in place.
#pragma once
#include <cstddef>
#include <cstdint>

namespace gbdmrg {

// A vector of `bytes` bytes of FP64 values at addr: it has to be device memory of the current
// device (device_memory), aligned as FP64 loads and stores need it, and to lie inside the allocation
// [base, base + size).  Everything else is copied, since a copy takes any alignment and turns
// an address that it cannot reach into an error, where a kernel would fault.
inline bool direct_vector(uintptr_t addr, size_t bytes, bool device_memory, uintptr_t base, size_t size) {
  return device_memory && addr % sizeof(double) == 0 && addr >= base && bytes <= size && addr - base <= size - bytes;
}

}  // namespace gbdmrg
