// bd_smem.h -- the dynamic shared-memory limits of the library's kernels
// (host only, no CUDA header: the device and the setter are passed in).
#pragma once

#include <cstddef>
#include <map>
#include <mutex>
#include <utility>

namespace bd {

// The limit is an attribute of a kernel on one device, so what has been set is
// remembered per device and kernel.  It only grows: launches planned for less
// stay valid, whatever plan, handle or thread asked for more since.
class SmemLimits {
  public:
    // Makes the limit at least `bytes`: set(fn, bytes) is called when this
    // device has not had as much for fn; its error is returned and forgets
    // nothing, so the next call tries again.
    template <typename Err, typename Set>
    Err raise(int dev, const void* fn, size_t bytes, Err ok, Set set)
    {
        std::lock_guard<std::mutex> lock(mu_);
        auto it = limit_.find({dev, fn});
        if (it != limit_.end() && it->second >= bytes) return ok;
        const Err e = set(fn, bytes);
        if (e == ok) limit_[{dev, fn}] = bytes;
        return e;
    }

  private:
    std::mutex mu_;
    std::map<std::pair<int, const void*>, size_t> limit_;
};

}  // namespace bd
