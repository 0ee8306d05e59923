// Setting something up once per device, from whichever threads come.
#pragma once
#include <atomic>
#include <mutex>

template <int DEVICES>
class SamOncePerDevice {
    std::atomic<bool> done_[DEVICES] = {};
    std::mutex mutex_;

public:
    // f() returns 0 if it succeeded; it runs again on the next call if it did not.  -1 for a device out of range.
    template <class F>
    int operator()(int device, F f) {
        if (device < 0 || device >= DEVICES) return -1;
        if (done_[device].load(std::memory_order_acquire)) return 0;
        std::lock_guard<std::mutex> lock(mutex_);
        if (done_[device].load(std::memory_order_relaxed)) return 0;
        const int rc = f();
        if (rc == 0) done_[device].store(true, std::memory_order_release);
        return rc;
    }
};
