// One-time preparation per device.
#pragma once

#include <cuda_runtime.h>

#include <mutex>

namespace tnbp {

// Kernel attributes (cudaFuncSetAttribute) belong to the current device, not to
// the process: they are set once for every device the library is used on.
class DeviceOnce {
 public:
  // The result of f(), run at the first call with this device current.
  template <class F>
  cudaError_t operator()(F f) {
    int dev = 0;
    const cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev < 0 || dev >= kMaxDevices) return f();
    std::call_once(once_[dev], [&] { result_[dev] = f(); });
    return result_[dev];
  }

 private:
  static constexpr int kMaxDevices = 64;
  std::once_flag once_[kMaxDevices];
  cudaError_t result_[kMaxDevices] = {};
};

}  // namespace tnbp
