// gs_device.cuh -- values that belong to a device: found once for each device of the process, by any thread.
// (A function attribute set on one device does not hold on another: the sort's 1024-thread kernel, whose runs need
// more shared memory than a launch gets unasked, was refused on every device but the first.)
#pragma once

#include <atomic>

namespace gs {

class PerDevice {
    static constexpr int kMaxDevices = 64;
    std::atomic<int> value[kMaxDevices] = {};   // 0: not found yet

public:
    // find() > 0, which is kept for device `dev`; 0 or less is a failure and asked for again
    template <class Find>
    int get(int dev, Find find) {
        if (dev < 0 || dev >= kMaxDevices) return find();
        int v = value[dev].load(std::memory_order_relaxed);
        if (v <= 0) {
            v = find();
            if (v > 0) value[dev].store(v, std::memory_order_relaxed);
        }
        return v;
    }
};

}  // namespace gs
