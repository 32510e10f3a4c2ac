// Something that is done once per device of the process: kernel attributes (shared memory beyond 48 KB, cluster sizes) belong to
// the device that is current when they are set, and a kernel that needs them does not start on another.
#pragma once
#include <mutex>

#include <cuda_runtime_api.h>

namespace jolt {

class DeviceOnce {
  std::once_flag flag_[64];

 public:
  template <typename F>
  void operator()(F &&set) {
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) set();
    else std::call_once(flag_[dev], set);
  }
};

}  // namespace jolt
