// dm_launch.h -- host-side launch arithmetic and state of the launchers.  No
// CUDA types: the host tests compile it too.
#pragma once

#include <atomic>
#include <cstddef>
#include <cstdint>
#include <mutex>

namespace dm {

constexpr int kDevices = 64;   // devices that per-device launch state is kept for

// The dynamic shared memory that one kernel (or kernels launched alike) has
// been allowed on each device.  The limit is a property of the kernel on a
// device, shared by every handle and thread, so it is only ever raised, under
// a lock: a smaller request that came later would lower it for a launch that
// another thread is about to make.
class SmemOptIn {
  public:
    // Makes sure `bytes` are allowed on device dev (0 <= dev < kDevices); set()
    // allows them and returns 0, or an error, which is returned.
    template <class Set>
    int raise(int dev, size_t bytes, Set set) {
        if (have_[dev].load(std::memory_order_acquire) >= bytes) return 0;
        std::lock_guard<std::mutex> lock(m_);
        if (have_[dev].load(std::memory_order_relaxed) >= bytes) return 0;
        const int e = set();
        if (!e) have_[dev].store(bytes, std::memory_order_release);
        return e;
    }

  private:
    std::mutex m_;
    std::atomic<size_t> have_[kDevices] = {};
};

// Trials per CTA (at most a warp's lanes) of the d-choices sweep, and its CTAs,
// such that every SM gets the same number of them: 10,000 trials on 152 SMs run
// as 3 x 152 CTAs of 22.
struct PotcShape {
    uint32_t per_cta, grid;
};
inline PotcShape potc_shape(uint64_t trials, uint64_t sms) {   // trials >= 1
    const uint64_t per_sm = (trials + sms * 32 - 1) / (sms * 32);
    const uint64_t T = (trials + sms * per_sm - 1) / (sms * per_sm);
    return {(uint32_t)T, (uint32_t)((trials + T - 1) / T)};
}

}  // namespace dm
