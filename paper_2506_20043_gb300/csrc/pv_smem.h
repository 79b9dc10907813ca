// pv_smem.h -- limits that launches look up and raise, shared by all host threads.
#pragma once
#include <atomic>
#include <mutex>

namespace pv {

constexpr int kMaxDevices = 64;

// A kernel's dynamic shared-memory limit per device. raise() sets it by set(bytes) (0 = done, else an error, which is
// returned) when a launch needs more than it was set to before, and never lowers it: threads that raise it at the
// same time set it one after the other, each only if the others have not set more. Otherwise a thread could set a
// smaller limit behind a larger one, and the launch that relies on that one would be refused.
class SmemLimit {
public:
    template <class Set>
    int raise(int device, int bytes, Set&& set) {
        if (bytes <= limit_[device].load(std::memory_order_acquire)) return 0;
        const std::lock_guard<std::mutex> hold(mutex_);
        if (bytes <= limit_[device].load(std::memory_order_relaxed)) return 0;
        const int e = set(bytes);
        if (e == 0) limit_[device].store(bytes, std::memory_order_release);
        return e;
    }

private:
    std::atomic<int> limit_[kMaxDevices] = {};
    std::mutex mutex_;
};

// Two properties of each device, looked up once by find(first, second) (0 = done): a thread that reads one sees both.
class DevicePair {
public:
    template <class Find>
    int get(int device, int& first, int& second, Find&& find) {
        first = first_[device].load(std::memory_order_acquire);
        if (first) {
            second = second_[device].load(std::memory_order_relaxed);
            return 0;
        }
        const int e = find(first, second);
        if (e) return e;
        second_[device].store(second, std::memory_order_relaxed);
        first_[device].store(first, std::memory_order_release);
        return 0;
    }

private:
    std::atomic<int> first_[kMaxDevices] = {}, second_[kMaxDevices] = {};
};

}  // namespace pv
