// device_once.cuh - set-up that holds for one device, made once on each (host code only).
#pragma once

#include <atomic>
#include <mutex>
#include <unordered_map>

namespace gr {

// The first call for a device runs f() and keeps its result; later calls return it.  Safe with several
// host threads; after the first call one atomic load for devices below kFast.
class DeviceOnce
{
public:
    template <class F>
    bool operator()(int device, F &&f)
    {
        const bool fast = device >= 0 && device < kFast;
        if (fast) {
            const int s = state_[device].load(std::memory_order_acquire);
            if (s) return s == kYes;
        }
        std::lock_guard<std::mutex> lock(mu_);
        auto it = done_.find(device);
        if (it == done_.end()) it = done_.emplace(device, f()).first;
        if (fast) state_[device].store(it->second ? kYes : kNo, std::memory_order_release);
        return it->second;
    }

private:
    static constexpr int kFast = 32, kYes = 1, kNo = 2;
    std::atomic<int> state_[kFast] = {};
    std::mutex mu_;
    std::unordered_map<int, bool> done_;
};

}  // namespace gr
