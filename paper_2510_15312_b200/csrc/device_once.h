// Set-up that a process needs once per device (function attributes, loading of kernels).
#pragma once
#include <atomic>

namespace sdv {

// Safe with several threads: the first ones may all run the set-up, which therefore has to bear repetition.  A set-up that failed
// is tried again by the next call; devices past the mask run it every time.
class DeviceOnce {
public:
    // `setup()` returns 0 for success; whatever it returns is handed back.
    template <typename F>
    auto run(int device, F setup) -> decltype(setup()) {
        const bool known = device >= 0 && device < 64;
        if (known && (done_.load(std::memory_order_acquire) >> device & 1ull)) return decltype(setup())(0);
        const auto rc = setup();
        if (known && (int)rc == 0) done_.fetch_or(1ull << device, std::memory_order_release);
        return rc;
    }

private:
    std::atomic<unsigned long long> done_{0};
};

}  // namespace sdv
