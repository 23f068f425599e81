// A limit of the process that only grows (a kernel attribute per device), raised by whichever thread
// needs more first. Plain host code, no CUDA.
#pragma once
#include <atomic>
#include <mutex>

namespace wmcd {

class RaisedLimit {
    std::atomic<int> have_{0};
    std::mutex m_;

  public:
    // Runs set(want) if the limit is below `want`; true when it is at least that afterwards. One thread at a
    // time, so a lower request never undoes a higher one; a request that set() refuses is not remembered.
    template <class F>
    bool raise(int want, F&& set) {
        if (want <= have_.load(std::memory_order_acquire)) return true;
        std::lock_guard<std::mutex> lock(m_);
        if (want <= have_.load(std::memory_order_relaxed)) return true;
        if (!set(want)) return false;
        have_.store(want, std::memory_order_release);
        return true;
    }
};

}  // namespace wmcd
