// What the SAP kernels (sap.cu, sap_apply.cu) share: the bounded wait for the
// bulk asynchronous copy of a domain's links.
#pragma once

#include "common.cuh"

namespace dwk {

__device__ __forceinline__ unsigned smem_u32(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }
__device__ __forceinline__ unsigned long long global_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}
// wait for a phase (by its parity) of the mbarrier, giving up after about a second
__device__ __forceinline__ bool bulk_copy_wait(unsigned long long* bar, unsigned parity = 0) {
    unsigned long long t0 = 0;
    for (unsigned it = 1;; ++it) {
        unsigned done;
        asm volatile(
            "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
            : "=r"(done)
            : "r"(smem_u32(bar)), "r"(parity)
            : "memory");
        if (done) return true;
        if ((it & 1023) == 0) {
            const unsigned long long now = global_ns();
            if (t0 == 0)
                t0 = now;
            else if (now - t0 > 1000000000ULL)
                return false;
        }
    }
}

}  // namespace dwk
