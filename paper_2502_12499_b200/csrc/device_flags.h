// Work done once per device: function attributes and occupancies belong to a device, and several threads may ask first.
#pragma once
#include <atomic>
#include <cstdint>

namespace ckpt {

constexpr int kMaxDevices = 64;

class DeviceFlags {
public:
    // set() for a device that has no successful call behind it; two threads may both run it.  0 = success.
    template <typename Set>
    int once(int device, Set&& set) {
        const bool known = device >= 0 && device < kMaxDevices;
        if (known && (done_.load(std::memory_order_acquire) >> device & 1u)) return 0;
        const int rc = set();
        if (rc == 0 && known) done_.fetch_or(uint64_t(1) << device, std::memory_order_release);
        return rc;
    }
    // The same for a value: find(out) fills it in, table[device] keeps it (written by one thread).
    template <typename Value, typename Find>
    int once(int device, Value* table, Value* out, Find&& find) {
        const bool known = device >= 0 && device < kMaxDevices;
        if (known && (done_.load(std::memory_order_acquire) >> device & 1u)) { *out = table[device]; return 0; }
        *out = Value();
        const int rc = find(out);
        if (rc == 0 && known && !(claimed_.fetch_or(uint64_t(1) << device) >> device & 1u)) {
            table[device] = *out;
            done_.fetch_or(uint64_t(1) << device, std::memory_order_release);
        }
        return rc;
    }

private:
    std::atomic<uint64_t> done_{0}, claimed_{0};
};

}  // namespace ckpt
