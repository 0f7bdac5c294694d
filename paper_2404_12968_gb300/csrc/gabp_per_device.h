// A value made once per device and kept for the life of the process, from any thread: launch limits,
// function attributes that have been set.  The first caller on a device makes it under a lock; once it
// is published, a call is one acquire load.  (Two plain statics, the device and the value, may be seen
// in either order by another thread: a grid of 0 blocks, then.)
#pragma once

#include <atomic>
#include <mutex>

namespace gabp {

template <typename V> class PerDevice {
    static constexpr int DEVICES = 64;   // beyond that the value is made on every call
    struct Slot {
        std::atomic<bool> ready{false};
        V value{};
    };
    Slot slot_[DEVICES];
    std::mutex mu_;

  public:
    // the value for device dev in out; make(out) forms it and returns an error code, 0 for success
    template <typename F> auto get(int dev, V &out, F make) -> decltype(make(out)) {
        using E = decltype(make(out));
        if (dev < 0 || dev >= DEVICES) return make(out);
        Slot &s = slot_[dev];
        if (!s.ready.load(std::memory_order_acquire)) {
            std::lock_guard<std::mutex> lock(mu_);
            if (!s.ready.load(std::memory_order_relaxed)) {
                const E e = make(s.value);
                if (e != E(0)) return e;
                s.ready.store(true, std::memory_order_release);
            }
        }
        out = s.value;
        return E(0);
    }
};

}  // namespace gabp
