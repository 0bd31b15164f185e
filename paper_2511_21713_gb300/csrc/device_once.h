// Work that has to be done once per device of the process: device symbols (constant tables) and kernel attributes
// belong to a device's context, and a mesh lives on whatever device is current.  Host only, no CUDA types.
#pragma once

#include <cstdint>
#include <mutex>

namespace pbfb {

class DeviceOnce {
 public:
  // f(), an int status with 0 for success, unless it has succeeded for this device; devices past the mask's 64 run
  // it each time.  Callers of one object wait for one another, so f is done for the device on return.
  template <class F>
  int run(int dev, F f) {
    std::lock_guard<std::mutex> lk(mu_);
    const bool kept = dev >= 0 && dev < 64;
    if (kept && ((done_ >> dev) & 1)) return 0;
    const int st = f();
    if (st == 0 && kept) done_ |= uint64_t(1) << dev;
    return st;
  }

 private:
  std::mutex mu_;
  uint64_t done_ = 0;
};

}  // namespace pbfb
