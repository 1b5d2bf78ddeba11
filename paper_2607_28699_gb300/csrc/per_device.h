// What a launch sets up once per device context of the process.  Function attributes belong
// to the context that was current when they were set, as do the answers of occupancy
// queries.  Host code only.
#pragma once

#include <atomic>
#include <mutex>

namespace wc {

// make(value) runs on the first get() in a device's context, and again while it returns an
// error or after the context was recreated; other calls, from any thread, find the value.  A
// device past kDevices, or a thread without a context yet (null), runs it each time.
template <typename T, typename Status = int>
class PerDevice {
public:
    static constexpr int kDevices = 64;

    template <typename Make>
    Status get(int device, const void* context, T& value, Make make) {
        if (device < 0 || device >= kDevices || !context) return make(value);
        Slot& s = slots_[device];
        if (s.context.load(std::memory_order_acquire) != context) {
            std::lock_guard<std::mutex> hold(mutex_);
            if (s.context.load(std::memory_order_relaxed) != context) {
                const Status st = make(s.value);
                if (st != Status{}) return st;
                s.context.store(context, std::memory_order_release);
            }
        }
        value = s.value;
        return Status{};
    }

private:
    struct Slot {
        std::atomic<const void*> context{nullptr};
        T value{};
    };
    Slot slots_[kDevices];
    std::mutex mutex_;
};

}  // namespace wc
