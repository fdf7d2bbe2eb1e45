// Something that the first user of a device does alone. Host code without CUDA, so that it can be tested by itself.
#pragma once

#include <mutex>
#include <vector>

namespace scw {

class FirstUse {
 public:
  // For a device without a successful first use, runs f() (its success is the result) while every other caller
  // waits here; otherwise returns at once. `ran`: f was called.
  template <typename F>
  bool alone(int device, bool& ran, F&& f) {
    std::lock_guard<std::mutex> lock(mu_);
    ran = false;
    for (int d : done_)
      if (d == device) return true;
    ran = true;
    if (!f()) return false;
    done_.push_back(device);
    return true;
  }

 private:
  std::mutex mu_;
  std::vector<int> done_;
};

}  // namespace scw
