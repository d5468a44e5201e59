// hoststage.h -- host staging of a call's list.  Plain C++ over an allocator of
// page-locked memory (a test exercises it without a GPU).
#pragma once

#include <algorithm>
#include <cstddef>
#include <cstdlib>
#include <cstring>

namespace f12host {

// Page-locked from kPinLeast to kPinMost bytes (copies run at the link's rate and
// need no intermediate copy: with the cores of plan_kinds 3.6 ms off a call of
// 200,000 quartets), plain memory below (the driver takes a small copy from plain
// memory 14 us sooner per call) and past that.  Grown on demand, given back
// with the context.  Pin: bool alloc(void **, size_t), void free(void *).
template <class Pin>
struct HostStage {
  static constexpr size_t kPinLeast = (size_t)256 << 10, kPinMost = (size_t)64 << 20;
  const bool may_pin;   // false: plain memory always (locking and unlocking pages stalls the device's other streams)
  unsigned char *p = nullptr;
  size_t cap = 0;
  bool pinned = false;
  explicit HostStage(bool pin) : may_pin(pin) {}
  bool reserve(size_t bytes, size_t keep = 0) {   // the first `keep` bytes stay
    if (bytes <= cap) return true;
    const size_t want = std::max(bytes + bytes / 4, (size_t)1 << 16);
    void *q = nullptr;
    const bool pin = may_pin && want >= kPinLeast && want <= kPinMost && Pin::alloc(&q, want);
    if (!pin) q = std::malloc(want);
    if (!q) return false;
    if (keep) std::memcpy(q, p, keep);
    release();
    p = (unsigned char *)q;
    cap = want;
    pinned = pin;
    return true;
  }
  void release() {
    if (pinned) Pin::free(p);
    else std::free(p);
    p = nullptr;
    cap = 0;
    pinned = false;
  }
};

}  // namespace f12host
