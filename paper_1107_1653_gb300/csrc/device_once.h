// Values found once per device (launch attributes set, occupancies looked up),
// in plain C++: kernel attributes belong to a device, and several threads may
// need them first at the same time.
#pragma once

#include <map>
#include <mutex>

namespace gs {

template <class T>
class PerDevice {
public:
    // The device's value, from init() at the first call for it; other threads wait
    // until it is complete.  Where init() throws, nothing is kept.
    template <class F>
    const T& get(int device, F&& init) {
        std::lock_guard<std::mutex> lk(mu_);
        auto it = values_.find(device);
        if (it == values_.end()) it = values_.emplace(device, init()).first;
        return it->second;
    }

private:
    std::mutex mu_;
    std::map<int, T> values_;
};

}  // namespace gs
