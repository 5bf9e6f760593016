// A positive number that is determined once per device, such as how many
// clusters of a kernel a device holds.  Determining it is also where a
// kernel's attributes are set, which belong to one device as well.
#pragma once

#include <atomic>

namespace sem3d {

struct PerDevice {
  static constexpr int kDevices = 64;
  std::atomic<int> value[kDevices] = {};

  // The number of device `device` into `out`: kept, or from `make(int& out)`,
  // whose status is returned (0: success).  Two threads may both call `make`
  // on first use.  Ordinals beyond the table are not kept.
  template <class Make>
  auto get(int device, int& out, Make make) -> decltype(make(out)) {
    const bool kept = device >= 0 && device < kDevices;
    out = kept ? value[device].load(std::memory_order_acquire) : 0;
    if (out > 0) return {};
    const auto status = make(out);
    if (kept && !status) value[device].store(out, std::memory_order_release);
    return status;
  }
};

}  // namespace sem3d
