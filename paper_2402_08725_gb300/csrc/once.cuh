// One-time set-up per device (internal, host code): kernel attributes, constant tables.
#pragma once

#include <atomic>
#include <mutex>

#include "common.cuh"

namespace sr {

// run(f): f() once on each device. Host threads making their first calls together wait for the one that
// does it; a set-up that failed is tried again by the next call.
class OncePerDevice {
  public:
    template <class F>
    sr_status run(F f) {
        int dev = 0;
        SR_CUDA(cudaGetDevice(&dev));
        return run_on(dev, f);
    }
    template <class F>
    sr_status run_on(int dev, F f) {
        const unsigned long long bit = dev < 64 ? 1ull << dev : 0ull;  // beyond: every call
        if (done.load(std::memory_order_acquire) & bit) return SR_OK;
        std::lock_guard<std::mutex> lock(m);
        if (done.load(std::memory_order_relaxed) & bit) return SR_OK;
        const sr_status st = f();
        if (st == SR_OK) done.fetch_or(bit, std::memory_order_release);
        return st;
    }

  private:
    std::mutex m;
    std::atomic<unsigned long long> done{0};
};

}  // namespace sr
