// Work done once per device for a key (no CUDA here, so that it can be tested without a GPU).
#pragma once

#include <algorithm>
#include <mutex>
#include <utility>
#include <vector>

namespace slr {

// A kernel's attributes, its dynamic shared-memory limit among them, belong to the device that
// was current when they were set: what was done for a key on one device says nothing of another.
class OncePerDevice {
public:
    // f() unless it has succeeded for (key, device) before; false (and not remembered) if f() fails.
    template <typename F>
    bool run(const void* key, int device, F f) {
        std::lock_guard<std::mutex> lk(mu_);
        const std::pair<const void*, int> k(key, device);
        if (std::find(done_.begin(), done_.end(), k) != done_.end()) return true;
        if (!f()) return false;
        done_.push_back(k);
        return true;
    }

private:
    std::mutex mu_;
    std::vector<std::pair<const void*, int>> done_;
};

}  // namespace slr
