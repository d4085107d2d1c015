// Values found or set once per device and key and kept for the process: a
// kernel's attributes and what the occupancy calculation says belong to one
// device.  Plain host code without CUDA calls, so that tests can use it with any
// device numbers.
#pragma once

#include <map>
#include <mutex>
#include <utility>

namespace mhs {

template <typename Key, typename Value>
class PerDevice {
public:
    // the value of key on this device, make()'s on first use; nothing is kept when
    // make throws, and threads that ask for it meanwhile wait
    template <typename F>
    Value get(int device, const Key& key, F&& make) {
        std::lock_guard<std::mutex> lk(mu_);
        const auto it = known_.find({device, key});
        if (it != known_.end()) return it->second;
        const Value v = make();
        known_.emplace(std::make_pair(device, key), v);
        return v;
    }

private:
    std::mutex mu_;
    std::map<std::pair<int, Key>, Value> known_;
};

}  // namespace mhs
