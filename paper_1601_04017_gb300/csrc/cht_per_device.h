// Numbers asked of the driver once per device and kept.  Host code alone,
// compiled without CUDA too.
#pragma once

#include <atomic>

namespace cht {

constexpr int kKeptDevices = 64;  // (devices beyond are asked every time)

// A number > 0 for each device.  `ask(&n)` answers for the current device,
// `dev`, and does whatever that device needs done before the number is used
// (kernel attributes are a device's own); it returns 0 or an error, which is
// not kept.
class PerDevice {
  public:
    template <typename Ask>
    auto get(int dev, int* n, Ask ask) -> decltype(ask(n)) {
        std::atomic<int>* const k = dev >= 0 && dev < kKeptDevices ? &kept_[dev] : nullptr;
        *n = k ? k->load(std::memory_order_acquire) : 0;
        if (*n > 0) return decltype(ask(n))(0);
        const auto e = ask(n);
        if (e == decltype(ask(n))(0) && k) k->store(*n, std::memory_order_release);
        return e;
    }

  private:
    std::atomic<int> kept_[kKeptDevices] = {};
};

}  // namespace cht
