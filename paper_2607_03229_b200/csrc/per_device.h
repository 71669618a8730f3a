// A number a device is asked for once.  Callers on several threads may ask at the same time; a query that fails (a result that is not
// positive) is made again by the next call instead of being kept for the life of the process.
#pragma once
#include <atomic>

namespace mpipe {

constexpr int kDevices = 64;   // beyond that, every call asks
struct PerDevice {
    std::atomic<int> value[kDevices] = {};
    template <typename Query>
    int get(int dev, Query&& query) {
        if (dev < 0) return 0;
        if (dev < kDevices) {
            const int known = value[dev].load(std::memory_order_relaxed);
            if (known > 0) return known;
        }
        const int n = query();
        if (n <= 0) return 0;
        if (dev < kDevices) value[dev].store(n, std::memory_order_relaxed);
        return n;
    }
};

}  // namespace mpipe
