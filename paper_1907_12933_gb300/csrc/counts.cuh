// counts.cuh -- a thread's counts over a part of a query's points, and their way into the
// query's 64-bit counters.
#pragma once
#include "dev.cuh"

namespace vbmc {

// Sum over the warp of 32-bit numbers, exact in 64 bits.
__device__ __forceinline__ unsigned long long warp_sum(unsigned v) {
    return ((unsigned long long)__reduce_add_sync(0xffffffffu, v >> 16) << 16) +
           __reduce_add_sync(0xffffffffu, v & 0xffffu);
}

struct PointCounts {
    unsigned adv = 0, pts = 0;        // the owner flushes before either can pass 2^32
    unsigned long long first = ~0ull;

    // The warp's counts into c (every lane calls it); the thread starts from zero again.
    __device__ __forceinline__ void flush(Counters* c) {
        const unsigned long long a = warp_sum(adv), p = warp_sum(pts);
        const bool lead = (threadIdx.x & 31) == 0;
        if (a) {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                const unsigned long long f = __shfl_xor_sync(0xffffffffu, first, o);
                first = f < first ? f : first;
            }
            if (lead) {
                atomicAdd(&c->n_adv, a);
                atomicMin(&c->first, first);
            }
        }
        if (p && lead) atomicAdd(&c->n_points, p);
        adv = pts = 0;
        first = ~0ull;
    }
};

}  // namespace vbmc
