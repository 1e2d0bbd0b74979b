// Work that has to be done once on each device (host side, plain C++).
#pragma once

#include <atomic>
#include <cstdint>

namespace jagg {

// Remembers the devices on which a call has succeeded.  Safe with several threads: run() returns
// success only after the call has succeeded on that device, by this thread or by another; two
// threads may both make it.  Devices past the 64th make it every time.
class OncePerDevice {
 public:
  // f() returns its status, whose zero value is success.
  template <class F>
  auto run(int device, F&& f) -> decltype(f()) {
    using Status = decltype(f());
    const uint64_t bit = device >= 0 && device < 64 ? uint64_t(1) << device : 0;
    if (done_.load(std::memory_order_acquire) & bit) return Status{};
    const Status st = f();
    if (st == Status{}) done_.fetch_or(bit, std::memory_order_release);
    return st;
  }

 private:
  std::atomic<uint64_t> done_{0};
};

}  // namespace jagg
