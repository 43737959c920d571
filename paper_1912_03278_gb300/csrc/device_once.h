// device_once.h -- what holds per device and is set or asked once for each: a kernel's
// shared-memory limit, the number of SMs.  Several threads may come first at
// the same time; each then does the work, which gives the same.
#pragma once
#include <atomic>
#include <cstdint>

namespace ihmc {

constexpr int ONCE_DEVICES = 64;   // devices beyond these are set up at every call

class DeviceOnce {
    std::atomic<uint64_t> done{0};

public:
    // set() on the first call for device dev that succeeds (returns its type's zero)
    template <class F>
    auto run(int dev, F set) -> decltype(set()) {
        const uint64_t bit = dev >= 0 && dev < ONCE_DEVICES ? 1ull << dev : 0ull;
        if (done.load() & bit) return decltype(set()){};
        const auto e = set();
        if (e == decltype(set()){}) done.fetch_or(bit);
        return e;
    }
};

class DeviceValue {
    std::atomic<int> v[ONCE_DEVICES] = {};

public:
    // ask() on the first call for device dev (0: no answer, asked again)
    template <class F>
    int get(int dev, F ask) {
        if (dev < 0 || dev >= ONCE_DEVICES) return ask();
        int x = v[dev].load();
        if (!x && (x = ask())) v[dev].store(x);
        return x;
    }
};

}  // namespace ihmc
