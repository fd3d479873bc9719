// Set-up that a device needs once (function attributes, constant tables), from any thread.
#pragma once
#include <mutex>

namespace ltmp2 {

// run(device, f): f() the first time a device is seen, under a lock (later callers wait for it and
// return at once).  f returns 0 on success; a failure is returned and not remembered, so that the next
// caller tries again.  Devices past the table run f every time.
class OncePerDevice {
 public:
  template <typename F> auto run(int device, F &&f) -> decltype(f()) {
    std::lock_guard<std::mutex> lock(mu_);
    const bool known = device >= 0 && device < kDevices;
    if (known && done_[device]) return decltype(f())(0);
    const auto e = f();
    if (known && e == decltype(f())(0)) done_[device] = true;
    return e;
  }

 private:
  static constexpr int kDevices = 64;
  std::mutex mu_;
  bool done_[kDevices] = {};
};

}  // namespace ltmp2
