// An answer that holds for a device, asked once for each: kernel attributes (larger shared
// memory, clusters of 16) are set on the function as the current device knows it, and what
// an occupancy query answers is that device's.
#pragma once
#include <atomic>

class PerDevice {
public:
    // ask() >= 0 for the device; two threads that come first at the same time both ask
    template <typename F>
    int get(int device, F ask) {
        if (device < 0 || device >= kDevices) return ask();
        int v = known_[device].load(std::memory_order_acquire);
        if (v == 0) {
            v = ask() + 1;
            known_[device].store(v, std::memory_order_release);
        }
        return v - 1;
    }

private:
    static constexpr int kDevices = 64;
    std::atomic<int> known_[kDevices] = {};   // the answer plus one, 0: not asked yet
};
