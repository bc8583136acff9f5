// One value per CUDA device (host code; plain C++, no CUDA headers).  A kernel's attributes and its occupancy belong to
// the device that was current when they were set or asked for: with one copy for the process, a handle on a second device
// launched kernels without the attribute that their shared memory needs.
#pragma once
#include <atomic>
#include <mutex>

namespace lbk {

template <class T>
class PerDevice {
    static constexpr int MAX = 64;
    std::mutex mu_;
    std::atomic<bool> have_[MAX] = {};  // val_ is written before, and not again
    T val_[MAX] = {};

  public:
    // *out: the value of device dev, made by make(T &) (0: success) the first time.  A failure's value is not kept.
    // Callable from any thread.
    template <class Make>
    int get(int dev, Make make, T *out) {
        if (dev < 0 || dev >= MAX) return make(*out);
        if (!have_[dev].load(std::memory_order_acquire)) {
            std::lock_guard<std::mutex> lock(mu_);
            if (!have_[dev].load(std::memory_order_relaxed)) {
                T v{};
                const int e = make(v);
                if (e != 0) return e;
                val_[dev] = v;
                have_[dev].store(true, std::memory_order_release);
            }
        }
        *out = val_[dev];
        return 0;
    }
};

}  // namespace lbk
