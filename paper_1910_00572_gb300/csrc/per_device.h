// What a launch sets up once per device (kernel attributes) and the number that comes out of it (the
// SM count, a cluster size), for host threads that launch at the same time: the number is published
// last and with release order, so a thread that sees it sees the set-up behind it.
#pragma once
#include <atomic>

namespace loc {

class PerDevice {
 public:
    // The number of device dev into *value; set_up(value) makes it (> 0) the first time.  Threads that
    // come first together each run set_up, which has to give the same every time.  Returns set_up's
    // error (0: none); nothing is kept of a set-up that failed or of devices past the last slot.
    template <typename F>
    auto get(int dev, int* value, F set_up) -> decltype(set_up(value)) {
        const bool kept = dev >= 0 && dev < kSlots;
        if (kept && (*value = v_[dev].load(std::memory_order_acquire)) > 0) return decltype(set_up(value))(0);
        const auto e = set_up(value);
        if (kept && e == decltype(set_up(value))(0)) v_[dev].store(*value, std::memory_order_release);
        return e;
    }

 private:
    static constexpr int kSlots = 64;
    std::atomic<int> v_[kSlots] = {};
};

}  // namespace loc
