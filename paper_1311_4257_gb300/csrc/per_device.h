// A value found out once per device, by whichever thread asks first; the others wait for it.
#pragma once
#include <mutex>
#include <stdexcept>

namespace dfmm {

template <class V>
class PerDevice {
 public:
  static constexpr int kDevices = 64;
  // find(): the value; if it throws, the next call asks again
  template <class F>
  V get(int dev, F&& find) {
    if (dev < 0 || dev >= kDevices) throw std::runtime_error("device ordinal out of range");
    std::call_once(once_[dev], [&] { v_[dev] = find(); });
    return v_[dev];
  }

 private:
  std::once_flag once_[kDevices];
  V v_[kDevices] = {};
};

}  // namespace dfmm
