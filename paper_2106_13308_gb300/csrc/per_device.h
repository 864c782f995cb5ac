// Set-up that a process does once for each device it uses, such as a kernel's limit
// of dynamic shared memory, which holds for the device that is current when it is
// set.  Any number of threads may call at the same time: more than one may then do
// the set-up, which has to allow that.  A failure is returned and not remembered.
#pragma once

#include <atomic>
#include <cstdint>

namespace vqmc {

class OncePerDevice {
 public:
  // f() returns 0 (cudaSuccess) when the set-up is done; beyond kDevices it is done on every call
  template <class F>
  auto operator()(int device, F f) -> decltype(f()) {
    const bool kept = device >= 0 && device < kDevices;
    const uint64_t bit = uint64_t(1) << (device & 63);
    if (kept && (done_[device / 64].load(std::memory_order_acquire) & bit)) return decltype(f())(0);
    const auto e = f();
    if (kept && e == decltype(f())(0)) done_[device / 64].fetch_or(bit, std::memory_order_release);
    return e;
  }

 private:
  static constexpr int kDevices = 256;
  std::atomic<uint64_t> done_[kDevices / 64] = {};
};

}  // namespace vqmc
