// What is looked up once per GPU and then read by every call: plain C++, compiled for the host in the CPU tests too.
#pragma once
#include <atomic>

namespace vla {

// A record per device.  The first call's thread looks it up; threads that come while it does so look it up for themselves, and one of
// them publishes its own, whole: a reader never sees a record that somebody is writing.  Nobody waits and nothing is thrown.
template <typename T>
class PerDevice {
 public:
  static constexpr int kMax = 64;
  // `look_up(T*)` fills a record or returns false (then nothing is kept and the next call tries again).
  template <typename F>
  bool get(int dev, T* out, F&& look_up) {
    if (dev < 0 || dev >= kMax) return false;
    Slot& s = slots_[dev];
    if (s.state.load(std::memory_order_acquire) == 2) { *out = s.value; return true; }
    T mine = T();
    if (!look_up(&mine)) return false;
    int empty = 0;
    if (s.state.compare_exchange_strong(empty, 1, std::memory_order_acquire)) {
      s.value = mine;
      s.state.store(2, std::memory_order_release);
    }
    *out = mine;
    return true;
  }

 private:
  struct Slot { std::atomic<int> state{0}; T value; };     // 0 empty, 1 being written, 2 published
  Slot slots_[kMax];
};

}  // namespace vla
