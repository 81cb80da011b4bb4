// Use of the caller's device arrays where they lie (internal header).
#pragma once
#include <cuda.h>
#include "common.cuh"

namespace tp {

using PointerQuery = CUresult (*)(unsigned, CUpointer_attribute*, void**, CUdeviceptr);

// Whether a kernel on `device` may use the caller's array: memory of that
// device, aligned to its type, `n` elements inside one allocation. A copy
// accepts any address (another GPU's too, which a kernel reaches only with peer
// access) and reports what it cannot reach, so everything else goes through one.
// With one device in the process all device memory is its own, and the query is
// spared the attribute (a third of a microsecond a pointer).
template <class T>
bool usable_in_place(PointerQuery query, int devices, int device, const T* p, size_t n) {
  const auto at = reinterpret_cast<uintptr_t>(p);
  if (!query || at % alignof(T)) return false;
  CUmemorytype type{};
  CUdeviceptr start = 0;
  size_t size = 0;
  int owner = devices > 1 ? -1 : device;
  CUpointer_attribute what[4] = {CU_POINTER_ATTRIBUTE_MEMORY_TYPE,
                                 CU_POINTER_ATTRIBUTE_RANGE_START_ADDR,
                                 CU_POINTER_ATTRIBUTE_RANGE_SIZE,
                                 CU_POINTER_ATTRIBUTE_DEVICE_ORDINAL};
  void* to[4] = {&type, &start, &size, &owner};
  return query(devices > 1 ? 4 : 3, what, to, at) == CUDA_SUCCESS && type == CU_MEMORYTYPE_DEVICE &&
         owner == device && at - start + n * sizeof(T) <= size;
}

}  // namespace tp
