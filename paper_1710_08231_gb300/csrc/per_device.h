// per_device.h -- values that belong to one device (a kernel's shared-memory limit and the blocks of it that fit an
// SM), found out once per device. Host code without CUDA headers.
#pragma once

#include <cstddef>
#include <map>
#include <mutex>
#include <tuple>

namespace gp {

// find(device, what, size, &value, make): the value of (device, what, size); `make(&value)` is called for the first
// request of each, and again for the next one if it returned other than 0. Returns make's status. Safe with several
// threads: a value is made once, and the others wait for it.
class PerDevice {
 public:
  template <class Make>
  int find(int device, const void *what, size_t size, int *value, Make make) {
    std::lock_guard<std::mutex> lk(mu_);
    const auto key = std::make_tuple(device, what, size);
    auto it = known_.find(key);
    if (it == known_.end()) {
      int v = 0;
      const int st = make(&v);
      if (st != 0) return st;
      it = known_.emplace(key, v).first;
    }
    *value = it->second;
    return 0;
  }

 private:
  std::mutex mu_;
  std::map<std::tuple<int, const void *, size_t>, int> known_;
};

}  // namespace gp
