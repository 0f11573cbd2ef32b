// Set-up of a kernel that belongs to one device (host).
#pragma once

#include <cuda_runtime_api.h>

#include <atomic>

namespace molt {

// A kernel's attributes (the shared-memory opt-in, cluster sizes) are set on one device's copy of it: get(init) runs
// init once on every device that a process launches the kernel on.  init returns a positive value, which is kept,
// or an error, which is returned and tried again by the next call.  Several threads may run init at once: it
// sets the same attributes.
class PerDevice {
  public:
    template <class F>
    int get(F init) {
        int dev = 0;
        if (cudaGetDevice(&dev) != cudaSuccess || dev < 0) return -1;
        if (dev >= kDevices) return init();
        int v = value_[dev].load(std::memory_order_acquire);
        if (v <= 0) {
            v = init();
            if (v > 0) value_[dev].store(v, std::memory_order_release);
        }
        return v;
    }

  private:
    static constexpr int kDevices = 64;
    std::atomic<int> value_[kDevices] = {};
};

}  // namespace molt
