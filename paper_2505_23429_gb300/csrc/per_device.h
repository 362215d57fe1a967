// Values that belong to a CUDA device (kernel attributes, answers of device queries), formed once
// per device of the process.  Host code only.
#pragma once
#include <mutex>
#include <stdexcept>

namespace a2 {

template <typename T>
class PerDevice {
 public:
  // The value of device `dev`, formed by init() at its first use there; an init() that throws
  // is run again at the next use.
  template <typename F>
  T at(int dev, F&& init) {
    if (dev < 0 || dev >= kMax) throw std::runtime_error("device index out of range");
    std::call_once(once_[dev], [&] { value_[dev] = init(); });
    return value_[dev];
  }

 private:
  static constexpr int kMax = 64;
  std::once_flag once_[kMax];
  T value_[kMax] = {};
};

}  // namespace a2
