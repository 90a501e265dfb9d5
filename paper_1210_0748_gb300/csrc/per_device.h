// Answers of the CUDA runtime that depend on a device and compiled code only,
// asked once per device and shared by the handles of all threads.
#pragma once

#include <atomic>

namespace kb {

struct PerDevice {
  static constexpr int kDevices = 64;
  std::atomic<int> known[kDevices] = {};  // 0 = not asked yet

  // The answer for `device`, from query() the first time.  A query that fails
  // returns 0, which is handed on but not kept: the next call asks again.
  // Threads that ask at the same time each query and store the same answer.
  template <typename Query>
  int get(int device, Query query) {
    if (device < 0 || device >= kDevices) return query();
    int v = known[device].load(std::memory_order_acquire);
    if (!v) {
      v = query();
      if (v > 0) known[device].store(v, std::memory_order_release);
    }
    return v;
  }
};

}  // namespace kb
