// What the host finds out once per device: function attributes, occupancy.
#pragma once

#include <mutex>

namespace sao {

// A value of each device, found by the first call that asks for it (a function
// attribute set on one device does not hold on another). Threads may ask at once;
// devices past the last slot are asked every time.
template <class T>
class PerDevice {
 public:
  template <class Find>
  T get(int device, Find find) {
    if (device < 0 || device >= kSlots) return find();
    std::call_once(once_[device], [&] { value_[device] = find(); });
    return value_[device];
  }

 private:
  static constexpr int kSlots = 64;
  std::once_flag once_[kSlots];
  T value_[kSlots] = {};
};

}  // namespace sao
