// Values that belong to a CUDA device, made at their first use on it: kernel
// attributes, SM counts and symbol addresses are a device's own, and a process
// may use several.
#pragma once

#include <map>
#include <mutex>

namespace mwi {

template <typename T>
class PerDevice {
    std::mutex mu;
    std::map<int, T> made;

public:
    // the value of device dev, from make() at the first call for that device; a
    // make() that throws leaves nothing behind, the next call tries again
    template <typename F>
    T get(int dev, F&& make) {
        std::lock_guard<std::mutex> lk(mu);
        auto it = made.find(dev);
        if (it == made.end()) it = made.emplace(dev, make()).first;
        return it->second;
    }
};

}  // namespace mwi
