// What a device answers (how many clusters of a kernel it co-schedules) and what is set on a device (a function
// attribute) belongs to that device: a process that uses several must not take the first one's answer for all.
#pragma once
#include <atomic>

namespace taskkv {

constexpr int kMaxDevices = 64;

// Answers to one question, kept per device and key (0 .. N - 1); zero-initialised, for use as a function-local static.
// ask() gives a number >= 0 and sets what the answer depends on for the current device, `dev`.  Threads may ask at the same
// time: they get the same answer.  A device number beyond the table is asked every time.
template <int N = 1>
struct PerDevice {
  std::atomic<int> answer[kMaxDevices][N];       // 0: not asked yet, otherwise the answer plus one

  template <class Ask>
  int get(int dev, int key, const Ask& ask) {
    if (dev < 0 || dev >= kMaxDevices) return ask();
    std::atomic<int>& a = answer[dev][key];
    int v = a.load(std::memory_order_acquire);
    if (v == 0) {
      v = ask() + 1;
      a.store(v, std::memory_order_release);
    }
    return v - 1;
  }
};

}  // namespace taskkv
