// The dynamic shared memory a kernel may be launched with, raised as launches ask
// for more.  Plain C++, so that it can be compiled and checked without a GPU.
#pragma once

#include <atomic>
#include <cstddef>
#include <map>
#include <mutex>

namespace zm {

// One per kernel (instance).  The attribute is process-wide and a launch may need
// any of several sizes, so two threads must never lower it for each other: it only
// grows, and is compared and set under one lock (a size seen by the unlocked look
// has been set before it was stored).
class SharedMemoryLimit {
    static constexpr size_t kEveryKernel = 32 * 1024;    // 48 KB with the static part need no attribute
    static constexpr int kFast = 64;
    std::atomic<size_t> seen_[kFast] = {};
    std::mutex mu_;
    std::map<int, size_t> set_;

  public:
    // `set(bytes)` sets the attribute on the current device, `dev`, and returns 0
    // or an error, which is passed on (and tried again by the next call).
    template <class Set>
    int raise(int dev, size_t bytes, Set set) {
        if (bytes <= kEveryKernel) return 0;
        const bool fast = dev >= 0 && dev < kFast;
        if (fast && bytes <= seen_[dev].load(std::memory_order_acquire)) return 0;
        std::lock_guard<std::mutex> lk(mu_);
        size_t& have = set_[dev];
        if (bytes <= have) return 0;
        const int e = set(bytes);
        if (e != 0) return e;
        have = bytes;
        if (fast) seen_[dev].store(bytes, std::memory_order_release);
        return 0;
    }
};

}  // namespace zm
