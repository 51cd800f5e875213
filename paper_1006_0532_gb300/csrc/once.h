// Work done once per device and safe with several host threads.
#pragma once

#include <atomic>

namespace pdfx {

// Kernel attributes belong to a function and a device, not to a context: they are set to the most
// that any launch needs, and a device counts as done only after they are set, so that no thread
// goes on to a launch before (threads that race set them twice, to the same values).  A setting
// that fails is tried again by the next caller.  A device out of range is never counted.
constexpr int kMaxDevices = 64;
struct OncePerDevice {
  std::atomic<bool> done[kMaxDevices] = {};
  // set(): 0 on success.  Returns 0 or set()'s error.
  template <typename F>
  int run(int device, F set) {
    const bool known = device >= 0 && device < kMaxDevices;
    if (known && done[device].load(std::memory_order_acquire)) return 0;
    const int rc = static_cast<int>(set());
    if (rc == 0 && known) done[device].store(true, std::memory_order_release);
    return rc;
  }
};

}  // namespace pdfx
