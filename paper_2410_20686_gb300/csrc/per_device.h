// A value that is worked out once per device of the process: kernel attributes belong to the device that was
// current when they were set, so a flag per process leaves every other device without them.
#pragma once
#include <atomic>

namespace odgs {

class PerDevice {
public:
    // make() > 0 is kept for the device; a failure (<= 0) is not, and the next call tries again. Threads that
    // meet here for the first time may each call make, which has to give them the same.
    template <class Make>
    int get(int device, Make make) {
        if (device < 0 || device >= kDevices) return make();
        int x = value_[device].load(std::memory_order_acquire);
        if (x <= 0 && (x = make()) > 0) value_[device].store(x, std::memory_order_release);
        return x;
    }

private:
    static constexpr int kDevices = 64;
    std::atomic<int> value_[kDevices] = {};
};

}  // namespace odgs
