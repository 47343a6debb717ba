// State that belongs to a device (function attributes, SM counts, occupancy),
// made once for each device of the process on its first use there.  Contexts on
// several devices may launch from several threads.
#pragma once

#include <mutex>

namespace dwfk {

template <class T, int N = 64>
class PerDevice {
 public:
  // make() runs once per device, with that device current.  Null beyond N
  // devices: the caller does without the cached state.
  template <class Make>
  const T* get(int dev, const Make& make) {
    if (dev < 0 || dev >= N) return nullptr;
    std::call_once(once_[dev], [&] { value_[dev] = make(); });
    return &value_[dev];
  }

 private:
  std::once_flag once_[N];
  T value_[N] = {};
};

}  // namespace dwfk
