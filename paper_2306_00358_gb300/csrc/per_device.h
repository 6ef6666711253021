// Work done once for every device of the process.
//
// A kernel's function attributes (the opt-in to more than 48 KB of dynamic
// shared memory) and its occupancy belong to a device, so a process-wide
// std::once_flag leaves the second GPU of a process without them.
#pragma once

#include <map>
#include <mutex>

namespace trg {

class PerDevice {
public:
    // f() of the first call for `device`, which has to be current.  If f
    // throws, the next call tries again.
    template <class F>
    int get(int device, F&& f) {
        std::lock_guard<std::mutex> lock(mu_);
        auto it = value_.find(device);
        if (it == value_.end()) it = value_.emplace(device, f()).first;
        return it->second;
    }

private:
    std::mutex mu_;
    std::map<int, int> value_;
};

}  // namespace trg
