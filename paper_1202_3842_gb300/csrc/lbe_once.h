// What has to happen once per device, from whichever thread comes first (no CUDA in here).
#pragma once
#include <atomic>

namespace lbe {

// once(device, f): runs f unless it has succeeded (returned 0) for this device before.  Two threads that come at
// the same time may both run it.
class PerDevice {
    std::atomic<unsigned long long> done{0};

  public:
    template <typename F>
    auto operator()(int device, F &&f) -> decltype(f()) {
        const unsigned long long bit = device >= 0 && device < 64 ? 1ull << device : 0ull;
        if (done.load(std::memory_order_acquire) & bit) return decltype(f()){};
        const auto r = f();
        if (r == decltype(f()){}) done.fetch_or(bit, std::memory_order_release);
        return r;
    }
};

}  // namespace lbe
