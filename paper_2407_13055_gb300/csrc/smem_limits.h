// Dynamic shared-memory limits of kernels, raised once where needed.
#pragma once
#include <cstddef>
#include <map>
#include <mutex>
#include <utility>

namespace ckks {

// The limit is an attribute of a kernel on a device, and setting it acts on the
// current device only: a process with contexts on several devices raises it on
// each. A limit that could not be raised is not recorded (the launch that needs
// it fails, and the next one asks again).
class SmemLimits {
 public:
  // Calls raise() (true: done) if kernel f's limit on the device is below bytes.
  template <class Raise>
  void at_least(int device, const void* f, size_t bytes, Raise raise) {
    std::lock_guard<std::mutex> lock(mu_);
    size_t& cur = done_[{device, f}];
    if (bytes > cur && raise()) cur = bytes;
  }

 private:
  std::mutex mu_;
  std::map<std::pair<int, const void*>, size_t> done_;
};

}  // namespace ckks
