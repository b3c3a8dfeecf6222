// What the library keeps per device: kernel attributes belong to a device's copy of a kernel, the SM count and the L2 window to
// the device itself.  Host code without any CUDA call, so that its bookkeeping can be tried out without devices.
#pragma once
#include <atomic>
#include <mutex>

namespace ssd {

// One T per device ordinal, set up at the first request for it.
template <typename T>
class DeviceTable {
public:
    static constexpr int kMax = 64;
    // The device's entry; `init(T &)` returns 0 once it has set it up (anything else is passed on, and it is tried again the
    // next time).  -1 for an ordinal outside the table.
    template <typename Init>
    int get(int dev, Init init, const T **out) {
        if (dev < 0 || dev >= kMax) return -1;
        Slot &s = slot_[dev];
        if (!s.ready.load(std::memory_order_acquire)) {
            std::lock_guard<std::mutex> lk(mu_);
            if (!s.ready.load(std::memory_order_relaxed)) {
                T v{};
                const int rc = init(v);
                if (rc) return rc;
                s.value = v;
                s.ready.store(true, std::memory_order_release);
            }
        }
        *out = &s.value;
        return 0;
    }

private:
    struct Slot {
        std::atomic<bool> ready{false};
        T value{};
    };
    Slot slot_[kMax];
    std::mutex mu_;
};

}  // namespace ssd
