// Bounded grid-wide barrier of the persistent cooperative kernels (the FIM
// solve, the multi-step solo Euler solver and the strip walks).
#pragma once
#include <cstdint>
#include <cstdlib>

namespace ripple {

// Default bound on the polls of a grid-barrier wait (several seconds).  The
// host may lower it (RIPPLE_GRID_SPIN_LIMIT) to exercise the timeout path.
constexpr uint32_t kGridSpinLimit = 1u << 26;

inline unsigned grid_spin_limit()
{
    unsigned limit = kGridSpinLimit;
    if (const char* lim = std::getenv("RIPPLE_GRID_SPIN_LIMIT")) {
        char* end = nullptr;
        const unsigned long v = std::strtoul(lim, &end, 10);
        if (end != lim && v < kGridSpinLimit) limit = (unsigned)v;
    }
    return limit;
}

// Grid barrier number b (1, 2, ...) of a launch over an arrival counter that
// only counts up (zero when the launch begins), with bounded polls.  Thread 0
// arrives with a release after the CTA barrier, so the CTA's stores precede
// it; its acquire and the second CTA barrier order the other CTAs' stores
// before every later load of this CTA.  sflag (shared memory) records a wait
// that ran out, and the call returns false from then on.
__device__ __forceinline__ bool grid_barrier(unsigned* count, unsigned b, unsigned spin_limit, int* sflag)
{
    __syncthreads();
    if (threadIdx.x == 0) {
        asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(count) : "memory");
        const unsigned target = b * gridDim.x;
        uint32_t i = 0;
        for (;;) {
            unsigned v;
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(count) : "memory");
            if ((int)(v - target) >= 0) break;
            if (++i > spin_limit) {
                sflag[0] = 1;
                break;
            }
        }
    }
    __syncthreads();
    return sflag[0] == 0;
}

}  // namespace ripple
