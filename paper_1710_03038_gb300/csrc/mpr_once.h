// A setting that holds per device (a kernel's shared-memory limit), made at most once on
// each, from any thread.
#pragma once

#include <atomic>
#include <cstdint>

namespace mpr {

class OncePerDevice {
public:
    // Runs set() unless it has succeeded (returned 0) on device dev before.  Two threads
    // may both run it, which does no harm; devices from 64 on always do.
    template <typename Set>
    auto operator()(int dev, Set set) -> decltype(set()) {
        const std::uint64_t bit = dev >= 0 && dev < 64 ? std::uint64_t{1} << dev : 0;
        if (done_.load(std::memory_order_acquire) & bit) return decltype(set()){};
        const auto status = set();
        if (status == decltype(set()){}) done_.fetch_or(bit, std::memory_order_release);
        return status;
    }

private:
    std::atomic<std::uint64_t> done_{0};
};

}  // namespace mpr
