// A setting that the CUDA runtime keeps per device, made once for each: plans on several
// devices, and threads, share a launcher.
#pragma once

#include <atomic>
#include <cstdint>

namespace dgm {

class OncePerDevice {
public:
    // true when the setting holds on `device`: calls `set` (returns true on success) the
    // first time, again after a failure, and always for devices past the 64 it remembers.
    // Two threads may both call `set`, which does no harm.
    template <typename F>
    bool ensure(int device, F&& set) {
        const uint64_t bit = device >= 0 && device < 64 ? uint64_t(1) << device : 0;
        if (done_.load(std::memory_order_acquire) & bit) return true;
        if (!set()) return false;
        done_.fetch_or(bit, std::memory_order_release);
        return true;
    }

private:
    std::atomic<uint64_t> done_{0};
};

}  // namespace dgm
