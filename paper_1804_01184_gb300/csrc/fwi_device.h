// fwi_device.h -- what is set up once per device (host only).
//
// Function attributes and occupancies belong to a device, not to the process: a value found on one
// device says nothing about another, and an attribute set there does not hold on another.
#pragma once
#include <map>
#include <mutex>

namespace fwi {

// make(dev), called once for each device, by one thread at a time.
template <class T>
class PerDevice {
public:
    template <class Make>
    T get(int dev, Make make)
    {
        std::lock_guard<std::mutex> lk(mu_);
        auto it = at_.find(dev);
        if (it == at_.end()) it = at_.emplace(dev, make(dev)).first;
        return it->second;
    }

private:
    std::mutex mu_;
    std::map<int, T> at_;
};

}  // namespace fwi
