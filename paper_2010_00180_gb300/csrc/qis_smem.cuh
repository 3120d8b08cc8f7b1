// qis_smem.cuh -- how much dynamic shared memory each kernel has been allowed, per device. The limit is a
// property of a kernel on a device, so what one context or network needs must not lower what another one's
// launch relies on, and a second device starts from nothing. (No CUDA header: tests compile it alone.)
#pragma once
#include <cstddef>
#include <map>
#include <mutex>
#include <utility>

namespace qis {

class SmemLimits {
 public:
  // set() raises the limit of `kernel` on device `dev` to `bytes`, where it has not been as much before;
  // returns its error (0: none, or nothing to do). Calls are made one at a time, so limits only grow.
  template <typename Set>
  int raise(int dev, const void* kernel, std::size_t bytes, Set set) {
    std::lock_guard<std::mutex> lock(mu_);
    std::size_t& have = have_[std::make_pair(dev, kernel)];
    if (bytes <= have) return 0;
    const int e = set();
    if (e == 0) have = bytes;
    return e;
  }

 private:
  std::mutex mu_;
  std::map<std::pair<int, const void*>, std::size_t> have_;
};

}  // namespace qis
