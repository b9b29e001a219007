// Set-up that CUDA keeps per device (a kernel's attributes, its occupancy), done before the first launch on each device.
#pragma once
#include <cuda_runtime.h>

#include <atomic>
#include <mutex>

namespace fwk {

// The value of f() on the current device, computed once per device.  A function-local static of this type does what a
// function-local static value does for a process that uses one device, and serves every other device as well.
template <class T>
class PerDevice {
    static constexpr int MAX = 64;
    std::mutex mu;
    std::atomic<bool> ready[MAX] = {};
    T value[MAX] = {};

public:
    template <class F>
    T get(F &&f)
    {
        int dev = -1;
        if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= MAX) return f();
        if (!ready[dev].load(std::memory_order_acquire)) {
            const std::lock_guard<std::mutex> lock(mu);
            if (!ready[dev].load(std::memory_order_relaxed)) {
                value[dev] = f();
                ready[dev].store(true, std::memory_order_release);
            }
        }
        return value[dev];
    }
};

}  // namespace fwk
