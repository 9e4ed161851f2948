// One-time kernel setup per device: function attributes (the shared-memory limit above 48 KiB) and
// occupancies belong to a device, not to the process.  Host only.
#pragma once

#include <mutex>

namespace svk {

template <typename T>
class PerDevice {
    static constexpr int MAX_DEVICES = 64;
    std::once_flag once_[MAX_DEVICES];
    T value_[MAX_DEVICES] = {};

public:
    // make()'s result for device dev, formed by the first call that asks for it (beyond
    // MAX_DEVICES: by every call).
    template <typename F>
    T get(int dev, F &&make) {
        if (dev < 0 || dev >= MAX_DEVICES) return make();
        std::call_once(once_[dev], [&] { value_[dev] = make(); });
        return value_[dev];
    }
};

}  // namespace svk
