// dwf_optin.h -- dynamic shared memory beyond 48 KB (host code, no CUDA types).
//
// A kernel has to be allowed more than 48 KB of dynamic shared memory before its first such
// launch, and the attribute that allows it belongs to the current device: a context on another
// GPU of the process needs its own.  One SmemOptIn per kernel remembers the largest size
// allowed so far on each device.
#pragma once

#include <cstddef>
#include <map>
#include <mutex>

namespace dwf {

constexpr size_t kSmemNoOptIn = 48 * 1024;

class SmemOptIn {
 public:
  // allow() raises the kernel's limit on the current device, `device`, and returns 0 on success;
  // it is called only where `bytes` is beyond what that device allows already.  Returns its
  // error, else 0.  Launches may come from several host threads.
  template <typename F>
  int ensure(int device, size_t bytes, F allow) {
    if (bytes <= kSmemNoOptIn) return 0;
    std::lock_guard<std::mutex> lock(mu_);
    size_t &have = allowed_[device];
    if (have >= bytes) return 0;
    const int e = allow();
    if (e == 0) have = bytes;
    return e;
  }

 private:
  std::mutex mu_;
  std::map<int, size_t> allowed_;
};

}  // namespace dwf
