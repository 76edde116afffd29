// device_once.h -- host work that is due once per device of the process (function attributes belong to the
// device that is current when they are set).
#pragma once
#include <cuda_runtime_api.h>

#include <mutex>

namespace isira {

// One static object per use; safe with several threads.  fn runs again on a device where it reported an error,
// and every time on devices beyond the 64 that are remembered.
class PerDeviceOnce {
public:
    template <class F>
    void operator()(F fn) {
        int dev = 0;
        if (cudaGetDevice(&dev) != cudaSuccess || dev < 0) return;   // the launch that follows reports it
        std::lock_guard<std::mutex> lock(mu_);
        if (dev < kDevices && done_[dev]) return;
        const bool ok = fn() == cudaSuccess;
        if (dev < kDevices) done_[dev] = ok;
    }

private:
    static constexpr int kDevices = 64;
    std::mutex mu_;
    bool done_[kDevices] = {};
};

}  // namespace isira
