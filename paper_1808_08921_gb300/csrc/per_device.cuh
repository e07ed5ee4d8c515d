// per_device.cuh -- a property of a device, found once in the process.
// Host code without kernels.
#pragma once
#include <mutex>

namespace lbmdem {

// Host threads that drive contexts of their own may ask at the same time: who
// asks while another is finding the value waits for it, so that all get the
// same.  Devices beyond the table have the value T{}.
template <class T, int DEVICES = 64>
class PerDevice {
    std::mutex mutex;
    bool known[DEVICES] = {};
    T value[DEVICES] = {};

public:
    template <class Find>
    T get(int dev, Find find) {
        if (dev < 0 || dev >= DEVICES) return T{};
        std::lock_guard<std::mutex> lock(mutex);
        if (!known[dev]) {
            value[dev] = find();
            known[dev] = true;
        }
        return value[dev];
    }
};

}  // namespace lbmdem
