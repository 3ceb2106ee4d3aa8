// An action taken once per device: a kernel's opt-in to more than 48 KB of
// dynamic shared memory holds on the device it was made on only.
#pragma once

#include <atomic>
#include <cstdint>

namespace shs {

class DeviceOnce {
public:
    // set() on the first call for `device` (and again after a failure); 0 is success.
    template <class F>
    auto run(int device, F&& set) -> decltype(set()) {
        const bool tracked = device >= 0 && device < 64;
        const uint64_t bit = tracked ? uint64_t{1} << device : 0;
        if (done_.load(std::memory_order_acquire) & bit) return decltype(set()){};
        const auto status = set();
        if (status == decltype(set()){}) done_.fetch_or(bit, std::memory_order_release);
        return status;
    }

private:
    std::atomic<uint64_t> done_{0};   // a bit per device
};

}  // namespace shs
