// Set-up that every device needs once per process (the dynamic shared memory limit
// of a kernel), for callers on several threads.
#pragma once

#include <stdint.h>
#include <atomic>
#include <mutex>

class HdDeviceOnce {
    std::atomic<uint64_t> done{0};
    std::mutex lock;

public:
    // Runs `set` (returning 0 or an error code) unless it has succeeded for `device`
    // before.  When this returns 0 it has: a thread that comes while another one is
    // at it waits, and one that comes after a failure tries again.
    template <class F>
    int run(int device, F set) {
        const uint64_t bit = 1ull << (device & 63);
        if (done.load(std::memory_order_acquire) & bit) return 0;
        std::lock_guard<std::mutex> hold(lock);
        if (done.load(std::memory_order_relaxed) & bit) return 0;
        const int rc = set();
        if (rc == 0) done.fetch_or(bit, std::memory_order_release);
        return rc;
    }
};
