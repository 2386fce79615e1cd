// A value that belongs to a device, found on the device's first use.
#pragma once

#include <mutex>

namespace tlr {

// Function attributes (shared-memory limit, cluster size) are set per device, and
// what they allow is a property of it: a flag kept once per process would skip
// them on every device but the first.  get(device, probe) runs probe, with that
// device current, once per device; other threads wait for it.
template <class T>
class PerDevice {
public:
    template <class F>
    T get(int device, F probe) {
        if (device < 0 || device >= kMax) return probe();
        std::lock_guard<std::mutex> lock(mu_);
        if (!known_[device]) {
            value_[device] = probe();
            known_[device] = true;
        }
        return value_[device];
    }

private:
    static constexpr int kMax = 64;
    std::mutex mu_;
    bool known_[kMax] = {};
    T value_[kMax] = {};
};

}  // namespace tlr
