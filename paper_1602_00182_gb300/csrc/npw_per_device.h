// npw_per_device.h -- state of a kernel's set-up that belongs to one device (its function attributes, its
// occupancy): one value per device, changed by one thread at a time.
#pragma once
#include <cuda_runtime.h>

#include <mutex>

namespace npw {

template <typename T>
class PerDevice {
public:
    // f(value of the current device) under the lock; on a device beyond the table f sees a fresh value
    // each time (the set-up is then repeated, which is harmless)
    template <typename F>
    cudaError_t with(F f) {
        int dev = 0;
        const cudaError_t e = cudaGetDevice(&dev);
        if (e != cudaSuccess) return e;
        if (dev < 0 || dev >= kDevices) {
            T fresh{};
            return f(fresh);
        }
        std::lock_guard<std::mutex> g(mu_);
        return f(val_[dev]);
    }
    // set() once per device, again after a failure
    template <typename F>
    cudaError_t once(F set) {
        return with([&](T& done) {
            if (done) return cudaSuccess;
            const cudaError_t e = set();
            done = e == cudaSuccess;
            return e;
        });
    }

private:
    static constexpr int kDevices = 64;
    std::mutex mu_;
    T val_[kDevices] = {};
};

}  // namespace npw
