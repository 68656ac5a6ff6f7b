// Set-up that belongs to a device (function attributes) rather than to the process.
#pragma once
#include <mutex>

namespace qc {

// Runs `set` once for each device and keeps its result for that device: one device's error is no other's, and threads on
// different devices share nothing.
template <typename Error>
class PerDevice {
 public:
  template <typename Set>
  Error once(int device, Set&& set) {
    Slot& s = slots_[device & 63];
    std::call_once(s.flag, [&] { s.error = set(); });
    return s.error;
  }

 private:
  struct Slot {
    std::once_flag flag;
    Error error{};
  };
  Slot slots_[64];
};

}  // namespace qc
