// Facts and settings of the current device (internal header).
#pragma once
#include <mutex>
#include "common.cuh"

namespace tp {

// devices that the process sees, at least 2 if the runtime cannot tell
inline int device_count() {
  static const int n = [] {
    int d = 0;
    return cudaGetDeviceCount(&d) == cudaSuccess ? d : 2;
  }();
  return n;
}

// make()'s value for the current device, made at the first call on it: kernel
// attributes and SM counts belong to a device, and a process may have contexts
// of the library on several. Safe with several threads; a make() that throws is
// tried again.
template <class T>
class PerDevice {
 public:
  template <class F>
  T operator()(F make) {
    int dev = 0;  // asked for where there is a choice: every launch of some kernels comes by
    if (device_count() != 1) TP_CUDA_TRY(cudaGetDevice(&dev));
    if (dev < 0 || dev >= kMax) return make();
    std::call_once(flag_[dev], [&] { value_[dev] = make(); });
    return value_[dev];
  }

 private:
  static constexpr int kMax = 64;
  std::once_flag flag_[kMax];
  T value_[kMax] = {};
};

// lets `kernel` take `bytes` of dynamic shared memory on the current device;
// `done` is a static of the caller's, one for each kernel
template <class K>
void allow_smem(PerDevice<bool>& done, K kernel, size_t bytes) {
  done([&] {
    TP_CUDA_TRY(cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     (int)bytes));
    return true;
  });
}

// SM count of the current device
inline int device_sms() {
  static PerDevice<int> sms;
  return sms([] {
    int dev = 0, v = 0;
    TP_CUDA_TRY(cudaGetDevice(&dev));
    TP_CUDA_TRY(cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, dev));
    return v;
  });
}

}  // namespace tp
