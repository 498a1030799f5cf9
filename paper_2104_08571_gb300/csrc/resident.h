// CTAs of a kernel that fit on an SM, with the kernel's opt-in to its dynamic
// shared memory.  Both belong to the current device: a context may be on any
// device, and the opt-in made on one says nothing about another, so the answer
// is kept per device.  A failure is not kept: the next call asks again.
#pragma once
#include <cuda_runtime.h>

#include <atomic>
#include <cstddef>

namespace ripple {

class ResidentCtas {
public:
    // 0 on error (which is cleared: it is not a later launch's)
    template <class K>
    int get(K kern, int threads, size_t smem)
    {
        int dev = -1, n = 0;
        if (cudaGetDevice(&dev) != cudaSuccess) return failed();
        std::atomic<int>* kept = dev >= 0 && dev < kDevices ? &kept_[dev] : nullptr;
        if (kept && (n = kept->load(std::memory_order_acquire)) > 0) return n;
        if (cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess ||
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kern, threads, smem) != cudaSuccess)
            return failed();
        if (kept && n > 0) kept->store(n, std::memory_order_release);
        return n;
    }

private:
    static int failed()
    {
        cudaGetLastError();
        return 0;
    }
    static constexpr int kDevices = 64;
    std::atomic<int> kept_[kDevices] = {};
};

}  // namespace ripple
