// What is found out, or set up, once per device, by whichever thread asks first.  Plain C++.
#pragma once
#include <atomic>

// A value for each device, T{} while it is not known.  Threads that ask before the first answer each work it out, and find the same.
template <typename T>
class PerDevice {
    std::atomic<T> known[64] = {};

public:
    // The value of device dev, from make() where it is not known; T{} where make() does not find one (the next call asks again).
    template <typename F>
    T get(int dev, F &&make) {
        if (dev < 0 || dev >= 64) return T{};
        T v = known[dev].load(std::memory_order_acquire);
        if (v == T{}) {
            v = make();
            if (v != T{}) known[dev].store(v, std::memory_order_release);
        }
        return v;
    }
};
