// bx_smem.h -- dynamic shared memory beyond the default limit (host side).
//
// cudaFuncAttributeMaxDynamicSharedMemorySize belongs to a kernel on one device, so the largest size
// set so far is kept per device: a process that uses a second device opts in there too, and threads
// that launch the same kernel with different sizes never lower it.
#pragma once

#include <stddef.h>

#include <mutex>

namespace bx {

class SmemOptIn {
  public:
    // Calls set(bytes) (0: success) unless that size or a larger one is set on the device; returns its
    // error, or 0.
    template <typename Set>
    int ensure(int device, size_t bytes, Set&& set) {
        std::lock_guard<std::mutex> lock(mu_);
        const bool known = device >= 0 && device < DEVICES;
        if (known && bytes <= size_[device]) return 0;
        const int e = set(bytes);
        if (known && e == 0) size_[device] = bytes;
        return e;
    }

  private:
    static constexpr int DEVICES = 64;   // beyond: set on every call
    std::mutex mu_;
    size_t size_[DEVICES] = {};
};

}  // namespace bx
