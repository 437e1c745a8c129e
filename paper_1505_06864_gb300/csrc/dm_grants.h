// Function attributes already raised, per device: an attribute such as the
// dynamic shared memory limit belongs to the device that is current when it is
// set, and plans may live on any device and be used from any thread.  Host
// code without CUDA.
#pragma once

#include <cstddef>
#include <map>
#include <mutex>
#include <utility>

namespace dm {

class Grants {
 public:
  // Calls set() unless `amount` or more was granted to `kernel` on `device`
  // before; what set() fails to raise (false) is asked for again next time.
  template <typename F>
  void ensure(int device, const void* kernel, size_t amount, F&& set) {
    std::lock_guard<std::mutex> lk(mu_);
    size_t& granted = granted_[std::make_pair(device, kernel)];
    if (amount > granted && set()) granted = amount;
  }

 private:
  std::mutex mu_;
  std::map<std::pair<int, const void*>, size_t> granted_;
};

}  // namespace dm
