// Kernel attributes that are set once per context.
//
// A block with more than 48 KB of dynamic shared memory needs
// cudaFuncAttributeMaxDynamicSharedMemorySize, and a kernel attribute holds
// for the device (the context on it) it was set for, not for the process.  So
// the record of what was set belongs to the library context, which has one
// device: a second context on another device sets its own.  Host code without
// CUDA headers, so that it is tested with a stand-in for the CUDA call.
#pragma once

#include <mutex>

namespace esplit {

class OptIn {
 public:
  // Runs set() the first time `kernel` is seen; 0, or what set() returned
  // (nothing is recorded then, and the next launch tries again).  Safe for
  // several threads on one context.
  template <class Set>
  int once(const void* kernel, Set set) {
    std::lock_guard<std::mutex> lock(m_);
    for (int k = 0; k < n_; ++k)
      if (done_[k] == kernel) return 0;
    if (const int rc = set()) return rc;
    if (n_ < CAP) done_[n_++] = kernel;  // beyond CAP kernels (several operator sizes): set again at each launch
    return 0;
  }

 private:
  static constexpr int CAP = 32;  // an operator size has at most 14 such kernels
  const void* done_[CAP] = {};
  int n_ = 0;
  std::mutex m_;
};

}  // namespace esplit
