// Values made once per device of the process: function attributes and device
// limits belong to the device that is current when they are set or asked.
#pragma once
#include <mutex>

namespace ibm {

template <class T>
class PerDevice {
 public:
  static constexpr int kDevices = 64;
  // the value of device dev, from make() on its first use (on every use beyond kDevices)
  template <class F>
  T get(int dev, F make) {
    if (dev < 0 || dev >= kDevices) return make();
    std::call_once(once_[dev], [&] { value_[dev] = make(); });
    return value_[dev];
  }

 private:
  std::once_flag once_[kDevices];
  T value_[kDevices]{};
};

}  // namespace ibm
