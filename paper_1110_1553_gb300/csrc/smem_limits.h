// Dynamic shared memory granted to the scheduler kernels so far. The limit is
// an attribute of a kernel on one device and must be raised before a launch
// that needs more; it is never lowered, as captured launches of other handles
// may rely on it. Plain C++ (no CUDA), without allocations.
#pragma once

#include <cstddef>
#include <mutex>

namespace hqr {

template <int Kernels, int Devices = 64>
class SmemLimits {
 public:
  // Calls set() if kernel slot `kernel` has not been granted `bytes` on device
  // `dev`; false if set() fails. Devices beyond the record are set every time.
  template <typename F>
  bool raise(int dev, int kernel, size_t bytes, F set) {
    if (dev < 0 || dev >= Devices) return set();
    std::lock_guard<std::mutex> lock(mutex_);  // held over set(): a smaller value never follows a larger one
    if (granted_[dev][kernel] >= bytes) return true;
    if (!set()) return false;
    granted_[dev][kernel] = bytes;
    return true;
  }

 private:
  std::mutex mutex_;
  size_t granted_[Devices][Kernels] = {};
};

}  // namespace hqr
