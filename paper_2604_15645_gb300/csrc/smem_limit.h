// Dynamic shared memory above what a launch gets unasked: which kernels' limits have been
// raised, and to what.
//
// cudaFuncSetAttribute raises a kernel's limit on the current device only, so the record is
// kept per handle (a handle belongs to one device, and to one context of it), not per
// process: the first call on a second device would be refused.  A limit is raised to all
// that the device offers beside the kernel's static memory, so handles that need different
// amounts do not lower each other's; a failure is not kept, the next call asks again.
// Host code without CUDA headers, so that it can be checked without a GPU.
#pragma once
#include <cstddef>

namespace pinn {

class SmemLimits {
 public:
  // Makes sure that `kern` may be launched with `bytes` of dynamic shared memory.
  // raise(&limit) raises its limit as far as the device allows and gives it, or an error;
  // `too_big` is returned when that is less than `bytes`.
  template <typename Err, typename Raise>
  Err allow(const void* kern, size_t bytes, Err ok, Err too_big, Raise&& raise) {
    for (int i = 0; i < n_; ++i)
      if (kern_[i] == kern) return bytes <= limit_[i] ? ok : too_big;
    size_t limit = 0;
    const Err e = raise(&limit);
    if (e != ok) return e;
    if (n_ < MAX) {   // (beyond that every call asks)
      kern_[n_] = kern;
      limit_[n_++] = limit;
    }
    return bytes <= limit ? ok : too_big;
  }

 private:
  static constexpr int MAX = 64;   // more than the kernels that one network reaches
  const void* kern_[MAX] = {};
  size_t limit_[MAX] = {};
  int n_ = 0;
};

}  // namespace pinn
