// bsp_smem.h -- the dynamic shared-memory limits that kernels have been given.
#pragma once

#include <stddef.h>

#include <atomic>
#include <mutex>

namespace bsp {

// A kernel's limit is an attribute of the kernel on one device, and setting it again
// lowers it as readily as it raises it.  One object per kernel (or per kernels with one
// size) keeps the limit of each device and only ever raises it: set() runs, under a lock, where
// the device has not got `bytes` yet, and a later smaller size asks for nothing.
class SmemLimit {
public:
    // set(bytes) returns an error code (0: done); devices past the table set it on every call.
    template <class Err, class Set>
    Err raise(int dev, size_t bytes, Set set) {
        const bool known = dev >= 0 && dev < DEVICES;
        if (known && at_[dev].load(std::memory_order_acquire) >= bytes) return Err(0);
        std::lock_guard<std::mutex> lock(mutex_);
        if (known && at_[dev].load(std::memory_order_relaxed) >= bytes) return Err(0);
        const size_t to = known || bytes > top_ ? bytes : top_;
        const Err e = set(to);
        if (e != Err(0)) return e;
        if (known) at_[dev].store(bytes, std::memory_order_release);
        else top_ = to;
        return Err(0);
    }

private:
    static constexpr int DEVICES = 64;
    std::mutex mutex_;
    std::atomic<size_t> at_[DEVICES] = {};
    size_t top_ = 0;   // the largest asked for on any device past the table
};

}  // namespace bsp
