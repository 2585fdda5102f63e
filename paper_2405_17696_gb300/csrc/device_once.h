// Work that is done once on every GPU of the process, e.g. a kernel's shared-memory limit:
// cudaFuncSetAttribute holds for the current device alone.  (No CUDA in here.)
#pragma once

#include <atomic>
#include <mutex>

namespace helm {

class DeviceOnce {
public:
    // set(), whose status 0 means success, unless it has succeeded on device `dev` before; its status.  A thread
    // that returns finds it done.  (Devices past the 64th run it every time.)
    template <class F>
    int run(int dev, F set) {
        const bool known = dev >= 0 && dev < 64;
        const unsigned long long bit = known ? 1ull << dev : 0ull;
        if (done_.load(std::memory_order_acquire) & bit) return 0;
        std::lock_guard<std::mutex> lk(mu_);
        if (done_.load(std::memory_order_relaxed) & bit) return 0;
        const int e = set();
        if (e == 0) done_.fetch_or(bit, std::memory_order_release);
        return e;
    }

private:
    std::mutex mu_;
    std::atomic<unsigned long long> done_{0};
};

}  // namespace helm
