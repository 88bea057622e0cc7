// launch.h -- host helpers for launches that depend on the device or context.
#pragma once

#include <cuda_runtime.h>

#include <atomic>

namespace mc {

// What a kernel needs set up on each device before its first launch there (an
// attribute of a function belongs to the device that is current): run at the
// first call on a device and at any later one until it succeeds.  Threads may
// run it side by side.
class OncePerDevice {
 public:
  template <typename F>
  bool operator()(F set_up) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0) return false;
    if (dev >= kDevices) return set_up();
    if (done_[dev].load(std::memory_order_acquire)) return true;
    if (!set_up()) return false;
    done_[dev].store(true, std::memory_order_release);
    return true;
  }

 private:
  static constexpr int kDevices = 128;
  std::atomic<bool> done_[kDevices] = {};
};

// A cooperative launch of at most `blocks` blocks, for a kernel that any grid
// will do for: where the stream's context holds fewer at once than the device
// (a partition of its SMs), the refused launch is repeated with half of them.
template <typename F>
cudaError_t launch_fitting(int blocks, F launch) {
  for (;; blocks /= 2) {
    const cudaError_t e = launch(blocks);
    if (e != cudaErrorCooperativeLaunchTooLarge || blocks <= 1) return e;
    cudaGetLastError();  // (the refusal is answered)
  }
}

}  // namespace mc
