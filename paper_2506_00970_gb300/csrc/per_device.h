// A value that is made once per device on its first use there: kernel
// attributes (a raised shared-memory limit, say) and occupancies belong to a
// device, so one made for the process would be missing, or wrong, on the
// second.  Host code without CUDA headers.
#pragma once

#include <mutex>

namespace gs2d {

constexpr int kMaxDevices = 64;

class PerDevice {
 public:
  // *value = the device's value, made by make(value) -- zero for success, else
  // the error that is returned, and the next call tries again.  Safe from
  // several threads.  Devices past the table make theirs at every call.
  template <class Make>
  int get(int device, int* value, Make make) {
    const std::lock_guard<std::mutex> lock(mu_);
    const bool kept = device >= 0 && device < kMaxDevices;
    if (kept && ready_[device]) {
      *value = value_[device];
      return 0;
    }
    const int err = make(value);
    if (err == 0 && kept) {
      value_[device] = *value;
      ready_[device] = true;
    }
    return err;
  }

 private:
  std::mutex mu_;
  bool ready_[kMaxDevices] = {};
  int value_[kMaxDevices] = {};
};

}  // namespace gs2d
