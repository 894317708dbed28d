// A value that belongs to a device (a kernel's attributes, its occupancy), set up
// by the first call made on that device.  Host code without CUDA, so that a CPU
// test can run it.
#pragma once

#include <mutex>

namespace qlin {

constexpr int kMaxDevices = 64;

template <typename T>
class PerDevice {
 public:
  // The value of device `dev` (0 <= dev < kMaxDevices), from make() the first
  // time; safe from several threads.
  template <typename F>
  const T& get(int dev, F&& make) {
    Slot& s = slots_[dev];
    std::call_once(s.once, [&] { s.value = make(); });
    return s.value;
  }

 private:
  struct Slot {
    std::once_flag once;
    T value{};
  };
  Slot slots_[kMaxDevices];
};

}  // namespace qlin
