// The devices a thread has prepared a kernel on (host only, no CUDA in this
// file).  Kernel attributes hold for one device, so a thread that drives a
// second device has to set them there as well.
#pragma once

namespace lstm_approx_impl {

class DeviceSet {
 public:
  bool has(int dev) const { return dev >= 0 && dev < 64 && (bits_ >> dev & 1ull) != 0; }
  void add(int dev) {  // devices from 64 on are not remembered: prepared on every launch
    if (dev >= 0 && dev < 64) bits_ |= 1ull << dev;
  }

 private:
  unsigned long long bits_ = 0;
};

}  // namespace lstm_approx_impl
