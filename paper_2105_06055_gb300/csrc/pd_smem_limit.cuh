// Dynamic shared-memory limits of kernels, as set so far (host only, private).
#pragma once

#include <cstddef>
#include <map>
#include <mutex>
#include <utility>

namespace pd {

// The limit belongs to a kernel function on a device, shared by every plan on that
// device and by every kernel node of a captured graph: it only ever grows, so plans
// of different sizes never lower it under each other. raise() calls set() where the
// recorded limit is below `bytes` and records what set() accepted; it returns set()'s
// status, 0 where nothing was to be set.
class SmemLimits {
public:
    template <class Set>
    int raise(int device, const void *func, size_t bytes, Set set)
    {
        std::lock_guard<std::mutex> lock(mu_);
        size_t &cur = limit_[{device, func}];
        if (bytes <= cur) return 0;
        const int e = set();
        if (e == 0) cur = bytes;
        return e;
    }

private:
    std::mutex mu_;
    std::map<std::pair<int, const void *>, size_t> limit_;
};

}  // namespace pd
