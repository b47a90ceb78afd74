// What a kernel needs set once on every device that it runs on.
#pragma once

#include <atomic>
#include <stdint.h>

namespace iqp {

// run(device, f): f() where it has not yet returned 0 for this device (always
// past the 64th); its error, or 0. Host threads that meet here may both call f.
struct DeviceOnce {
    std::atomic<uint64_t> done{0};

    template <class F>
    int run(int device, F f) {
        const uint64_t bit = device >= 0 && device < 64 ? (uint64_t)1 << device : 0;
        if (done.load(std::memory_order_acquire) & bit) return 0;
        const int e = f();
        if (e == 0) done.fetch_or(bit, std::memory_order_release);
        return e;
    }
};

}  // namespace iqp
