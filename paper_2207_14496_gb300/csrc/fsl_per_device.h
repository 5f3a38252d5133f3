// A launch parameter that is found once per device: the grid of a kernel whose
// blocks are all resident at once, or that a kernel's opt-in to large shared
// memory has been made.  Both hold for the device that was current, so a
// process with handles on several devices needs one of each per device.
// (Plain C++, no CUDA.)
#pragma once
#include <atomic>

namespace fsl {

class PerDevice {
 public:
  static constexpr int kDevices = 64;  // devices beyond are asked every time
  // The number of device dev, or make(&number)'s answer (number > 0, status
  // 0 for success) where none is kept yet.  A failure is returned and not
  // kept.  Threads that come first together may all call make.
  template <class Status, class Make>
  Status get(int dev, int* number, Make&& make, Status ok) {
    const bool keep = dev >= 0 && dev < kDevices;
    if (keep) {
      *number = kept_[dev].load(std::memory_order_acquire);
      if (*number > 0) return ok;
    }
    const Status s = make(number);
    if (s == ok && keep) kept_[dev].store(*number, std::memory_order_release);
    return s;
  }

 private:
  std::atomic<int> kept_[kDevices] = {};
};

}  // namespace fsl
