// lbm_once.h -- a set-up that is done once on each device (a kernel's function attributes).  Host
// code only.
#pragma once

#include <stdint.h>

#include <atomic>
#include <mutex>

namespace lbm {

// Function attributes belong to the kernel and the device, shared by every handle of the
// process, and handles may be stepped by several host threads: whatever sets them has to set them to
// one value, before the first launch that needs it, and never again.
class OncePerDevice {
    std::mutex lock_;
    std::atomic<uint64_t> done_{0};   // bit d: device d is set up

public:
    // set() returns 0 or an error; after an error the next call tries again.  When run() returns 0,
    // set() has been completed on `device`, by this thread or another one.
    template <typename Set> int run(int device, Set set)
    {
        const uint64_t bit = device >= 0 && device < 64 ? uint64_t(1) << device : 0;   // (others: every time)
        if (done_.load(std::memory_order_acquire) & bit) return 0;
        std::lock_guard<std::mutex> guard(lock_);
        if (done_.load(std::memory_order_relaxed) & bit) return 0;
        const int e = set();
        if (e == 0) done_.fetch_or(bit, std::memory_order_release);
        return e;
    }
};

}  // namespace lbm
