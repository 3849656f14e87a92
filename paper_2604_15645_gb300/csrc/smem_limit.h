// Dynamic shared memory above what a launch gets unasked: which kernels' limits have been
// raised, and to what.
//
// cudaFuncSetAttribute raises a kernel's limit in the current device's context only, so a
// record belongs to one context, never to the process: the first call on a second device
// would be refused.  The handles of a context share its record (a network family's 64 handles
// raise each limit once, not 64 times: 0.5 ms of its first step).  A limit is raised to all
// that the device offers beside the kernel's static memory, so handles that need different
// amounts do not lower each other's; a failure is not kept, the next call asks again.
// Host code without CUDA headers, so that it can be checked without a GPU.
#pragma once
#include <atomic>
#include <cstddef>
#include <cstdint>
#include <mutex>

namespace pinn {

class SmemLimits {
 public:
  // Makes sure that `kern` may be launched with `bytes` of dynamic shared memory.
  // raise(&limit) raises its limit as far as the device allows and gives it, or an error;
  // `too_big` is returned when that is less than `bytes`.  From any thread: entries are only
  // added, and two threads that raise the same limit raise it to the same value.
  template <typename Err, typename Raise>
  Err allow(const void* kern, size_t bytes, Err ok, Err too_big, Raise&& raise) {
    for (int i = 0, n = n_.load(std::memory_order_acquire); i < n; ++i)
      if (kern_[i] == kern) return bytes <= limit_[i] ? ok : too_big;
    size_t limit = 0;
    const Err e = raise(&limit);
    if (e != ok) return e;
    std::lock_guard<std::mutex> lock(add_);
    const int n = n_.load(std::memory_order_relaxed);
    bool known = false;   // (another thread was faster)
    for (int i = 0; i < n; ++i) known = known || kern_[i] == kern;
    if (!known && n < MAX) {   // (beyond that every call asks)
      kern_[n] = kern;
      limit_[n] = limit;
      n_.store(n + 1, std::memory_order_release);
    }
    return bytes <= limit ? ok : too_big;
  }

 private:
  static constexpr int MAX = 128;   // more than the library's kernels
  const void* kern_[MAX] = {};
  size_t limit_[MAX] = {};
  std::atomic<int> n_{0};
  std::mutex add_;
};

// The records of the contexts seen so far, by the id that the driver never gives twice.
class ContextLimits {
 public:
  // The context's record; nullptr once MAX contexts have been seen (a program that resets its
  // device again and again): the caller then keeps a record of its own.
  SmemLimits* of(uint64_t context) {
    std::lock_guard<std::mutex> lock(add_);
    for (int i = 0; i < n_; ++i)
      if (context_[i] == context) return &limits_[i];
    if (n_ == MAX) return nullptr;
    context_[n_] = context;
    return &limits_[n_++];
  }

 private:
  static constexpr int MAX = 32;
  uint64_t context_[MAX] = {};
  SmemLimits limits_[MAX];
  int n_ = 0;
  std::mutex add_;
};

}  // namespace pinn
