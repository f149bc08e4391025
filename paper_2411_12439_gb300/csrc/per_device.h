// A value that is made once for each device, at its first use there: launch limits and
// attributes of a kernel, which CUDA keeps per device.  Contexts of several devices
// and host threads may share one; a failure is not kept, so the next use tries again.
#pragma once

#include <atomic>
#include <mutex>

namespace lcg {

constexpr int kMaxDevices = 256;

template <typename T>
class PerDevice {
public:
    // out = the value of `device`; `make(T&)` makes it and returns 0 (of any error
    // type) or why it could not, which is then returned.
    template <typename Make>
    auto get(int device, T& out, Make make) -> decltype(make(out)) {
        using Err = decltype(make(out));
        if (device < 0 || device >= kMaxDevices) return make(out);
        Entry& e = entry_[device];
        if (!e.ready.load(std::memory_order_acquire)) {
            std::lock_guard<std::mutex> lock(mu_);
            if (!e.ready.load(std::memory_order_relaxed)) {
                T v{};
                const Err err = make(v);
                if (err != Err{}) return err;
                e.value = v;
                e.ready.store(true, std::memory_order_release);
            }
        }
        out = e.value;
        return Err{};
    }

private:
    struct Entry {
        std::atomic<bool> ready{false};
        T value{};
    };
    std::mutex mu_;
    Entry entry_[kMaxDevices];
};

}  // namespace lcg
