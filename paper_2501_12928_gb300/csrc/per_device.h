// What holds for one device only (a kernel's shared memory allowance, the number of
// SMs, the clusters that fit) is formed once for each device that is used.
#pragma once

#include <cuda_runtime.h>

#include <map>
#include <mutex>

namespace beor {

template <typename T>
class PerDevice {
 public:
  // the current device's value, from make() at its first use there
  template <typename F>
  T get(F make) {
    int device = 0;
    cudaGetDevice(&device);
    std::lock_guard<std::mutex> lk(mu_);
    auto it = values_.find(device);
    if (it == values_.end()) it = values_.emplace(device, make()).first;
    return it->second;
  }

 private:
  std::mutex mu_;
  std::map<int, T> values_;
};

// Internal linkage below: each build of the library in a process has its own kernels.
// SMs of the current device
static inline int device_sms() {
  static PerDevice<int> sms;
  return sms.get([] {
    int device = 0, n = 0;
    cudaGetDevice(&device);
    return cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, device) == cudaSuccess && n > 0 ? n : 1;
  });
}
// Allows kernel `kern` `bytes` of dynamic shared memory on the current device.
template <auto kern>
static cudaError_t allow_smem(int bytes) {
  static PerDevice<cudaError_t> done;
  return done.get([&] { return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes); });
}

}  // namespace beor
