// once_per_device.cuh -- host code that has to have run once for each device, such
// as a kernel's shared-memory limit, which the runtime keeps per device: a
// process that builds on a second GPU needs it set there as well.
#pragma once

#include <atomic>
#include <cstdint>

namespace lbvh {

class OncePerDevice {
public:
    // Runs f() unless it has succeeded for device `dev` before; false if it
    // fails now (it then runs again the next time). Threads may call this
    // together: each returns after a run that succeeded, its own or another's.
    template <typename F>
    bool operator()(int dev, F &&f) {
        const uint64_t bit = dev >= 0 && dev < 64 ? uint64_t(1) << dev : 0;  // others: every time
        if (done_.load(std::memory_order_acquire) & bit) return true;
        if (!f()) return false;
        done_.fetch_or(bit, std::memory_order_release);
        return true;
    }

private:
    std::atomic<uint64_t> done_{0};
};

}  // namespace lbvh
