// Work done once for each device by whichever thread comes first.
#pragma once

#include <atomic>
#include <cstdint>

namespace cube2 {

// Function attributes (the opt-in to more than 48 KB of dynamic shared memory) belong
// to a kernel on one device.  A failed attempt is not remembered; two threads that come
// at once both make it, which does no harm.
class PerDevice {
    std::atomic<uint64_t> done{0};

public:
    // f() on this device's first call (every call from the 65th device on); f returns 0 if it worked
    template <class F>
    auto once(int device, F f) -> decltype(f()) {
        const uint64_t bit = device >= 0 && device < 64 ? 1ull << device : 0;
        if (done.load(std::memory_order_acquire) & bit) return decltype(f())(0);
        const auto e = f();
        if (e == decltype(f())(0)) done.fetch_or(bit, std::memory_order_release);
        return e;
    }
};

}  // namespace cube2
