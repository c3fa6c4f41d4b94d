// fem_wait.cuh -- the bounded wait of the solves' loop kernel at its grid barrier.
#pragma once

#include <stdint.h>

#include "fem_internal.cuh"

namespace fem {

// One thread waits until the counter *p has reached `target` (modulo 2^32); what other CTAs wrote
// before they raised it is visible afterwards. After budget_ns (%globaltimer, looked at every 256
// reads) it sets *gave_up, records a timeout in *err and returns false.
__device__ __forceinline__ bool wait_reached(const unsigned *p, unsigned target, uint64_t budget_ns, unsigned *gave_up,
                                             unsigned *err) {
    uint64_t t0 = 0, t = 0;
    unsigned spins = 0;
    for (;;) {
        unsigned seen;
        asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(seen) : "l"(p) : "memory");
        if (static_cast<int>(seen - target) >= 0) return true;
        if ((++spins & 255u) == 0u) {
            asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
            if (t0 == 0) t0 = t;
            if (t - t0 > budget_ns) {
                atomicExch(gave_up, 1u);
                record_device_error(err, FEM_DEVERR_TIMEOUT);
                return false;
            }
        }
    }
}

}  // namespace fem
