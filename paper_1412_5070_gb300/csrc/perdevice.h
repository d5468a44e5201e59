// perdevice.h -- values that a process holds once per device (constant tables
// and the addresses of what was allocated for them).  Plain C++ (a test
// exercises it without a GPU).
#pragma once

#include <map>
#include <mutex>

namespace f12host {

template <class T>
class PerDevice {
 public:
  // The device's value, made by fill(T &) at its first use; fill returns 0, or a
  // status that is passed on (the next call tries again).
  template <class Fill>
  int get(int device, T *out, Fill fill) {
    std::lock_guard<std::mutex> lk(mu_);
    auto it = value_.find(device);
    if (it == value_.end()) {
      T v{};
      const int rc = fill(v);
      if (rc != 0) return rc;
      it = value_.emplace(device, v).first;
    }
    *out = it->second;
    return 0;
  }

 private:
  std::mutex mu_;
  std::map<int, T> value_;
};

}  // namespace f12host
