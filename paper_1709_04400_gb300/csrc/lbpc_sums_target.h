// Where the domain-sum reduction may write a caller's two doubles itself, instead of a copy after it. Host code without
// device parts, so that a host compiler can build it by itself.
#pragma once

#include <stdint.h>

#include <initializer_list>

#include <cuda_runtime_api.h>

namespace lbpc {

// What the runtime and the driver say of one address: its attributes, the access of the current device
// (CU_POINTER_ATTRIBUTE_ACCESS_FLAGS; 3: reads and writes), and the end of its allocation (0 if unknown).
struct AddressInfo {
  cudaPointerAttributes at;
  unsigned long long access;
  uintptr_t past;
};

// The address under which a kernel on `device` writes out[0] and out[1], or null where a copy must do it, which checks
// what it is given: memory of the other kind than on_device says, another device's, managed or pageable memory, memory
// that the device may not write or that ends within the 16 bytes (first, last: of their first and last byte).
inline double* sums_target(double* out, bool on_device, int device, const AddressInfo& first, const AddressInfo& last) {
  const cudaMemoryType want = on_device ? cudaMemoryTypeDevice : cudaMemoryTypeHost;
  if (((uintptr_t)out & 7) != 0) return nullptr;
  for (const AddressInfo* a : {&first, &last})
    if (a->at.type != want || (on_device && a->at.device != device) || (a->access & 3) != 3) return nullptr;
  char* p = (char*)first.at.devicePointer;
  if (!p || (char*)last.at.devicePointer != p + 2 * sizeof(double) - 1) return nullptr;
  return (double*)p;
}

}  // namespace lbpc
