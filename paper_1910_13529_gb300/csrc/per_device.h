// What a launch has set up, per device: plain C++.
#pragma once

#include <atomic>
#include <mutex>

namespace pic {

// A kernel's shared-memory limit belongs to the device that is current when it is set.  One of these beside
// each kernel's launch keeps what each device has been granted; handles on several devices and threads
// that launch at once share it.
class PerDevice {
  public:
    // set(amount), unless the device already has that much: 0, or the error of set.  Grants only grow.
    template <typename F>
    int grant(int device, int amount, F&& set) {
        const bool known = device >= 0 && device < N;
        if (known && have_[device].load(std::memory_order_acquire) >= amount) return 0;
        std::lock_guard<std::mutex> lock(m_);
        if (known && have_[device].load(std::memory_order_relaxed) >= amount) return 0;
        const int e = set();
        if (e == 0 && known) have_[device].store(amount, std::memory_order_release);
        return e;
    }

    // the number make() gives for the device, asked for once (again while it is 0)
    template <typename F>
    int number(int device, F&& make) {
        const bool known = device >= 0 && device < N;
        int v = known ? have_[device].load(std::memory_order_acquire) : 0;
        if (v == 0) {
            v = make();
            if (known) have_[device].store(v, std::memory_order_release);
        }
        return v;
    }

  private:
    static constexpr int N = 64;           // beyond: set up at every launch
    std::atomic<int> have_[N] = {};
    std::mutex m_;
};

}  // namespace pic
