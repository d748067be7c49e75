// Dynamic shared-memory limits of kernels.  A kernel's limit above 48 KB is an attribute of the
// kernel on one device: one process may use several, from several threads.
#pragma once
#include <cstddef>
#include <map>
#include <mutex>
#include <utility>

namespace kpcg {

class SmemLimits {
public:
    // Calls set(), which raises the limit of `kern` on device `dev` to `bytes`, unless it
    // stands at `bytes` or more there.  A set() that throws is tried again next time.
    template <typename Set>
    void allow(int dev, const void* kern, size_t bytes, Set&& set) {
        std::lock_guard<std::mutex> lock(mutex_);
        size_t& have = done_[{dev, kern}];
        if (bytes <= have) return;
        set();
        have = bytes;
    }

private:
    std::mutex mutex_;
    std::map<std::pair<int, const void*>, size_t> done_;
};

}  // namespace kpcg
