// One T per device, created on first use: function attributes, and what was found
// of a kernel's residency, belong to the device they were set or probed on, and a
// process may go on to another one.  Safe from several threads; the reference stays
// valid.
#pragma once

#include <cuda_runtime.h>

#include <map>
#include <mutex>

namespace ifmm {

template <class T>
class PerDevice {
  std::mutex mu_;
  std::map<int, T> v_;

 public:
  T& operator()() {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) cudaGetLastError();
    std::lock_guard<std::mutex> lock(mu_);
    return v_[dev];
  }
};

}  // namespace ifmm
