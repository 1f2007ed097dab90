// What the library keeps once for each GPU of the process: limits of kernels, the SM count, flags
// in device memory.  (A function's attributes belong to the device that is current when they are
// set: kept for the whole process, they are missing on the second GPU.)
#pragma once
#include <mutex>

namespace lddmm {

constexpr int kKeptDevices = 64;

// A value made on the first use with each device.  T{} stands for "none": a device whose make()
// returned it is tried again at the next use.  Devices past kKeptDevices get a new one every time.
template <typename T>
class PerDevice {
 public:
  template <typename Make>
  T get(int device, Make make) {
    if (device < 0 || device >= kKeptDevices) return make();
    std::lock_guard<std::mutex> hold(lock_);
    if (value_[device] == T{}) value_[device] = make();
    return value_[device];
  }

 private:
  std::mutex lock_;
  T value_[kKeptDevices] = {};
};

}  // namespace lddmm
