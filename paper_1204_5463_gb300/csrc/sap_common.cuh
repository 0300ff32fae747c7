// Building blocks of the SAP kernels (sap.cu, sap_apply.cu): the shared-memory
// layouts of a domain's links and of the MR iterate, the CTA-wide sums of an MR
// step, and the bulk asynchronous copy of a domain's link image.
#pragma once

#include "common.cuh"

namespace dwk {

// The domain's own links in shared memory, packed so that one link matrix
// (9 complex entries) is read with as few wide loads as possible:
//   P64      double2 [4][9][T]                                          (9 x 16 B loads)
//   P32      float2 [4][9][T]                                           (9 x 8 B loads)
//   P16/B16  uint4 [4][2][T] (entry quads) + uint32 [4][T] (entry 8)    (2 x 16 B + 4 B)
// pack() writes that layout for one site of a domain into a global image of
// the domain (built once per gauge field), so that a CTA stages all its links
// with one bulk asynchronous copy. (FP32 entry pairs packed as float4
// measured no faster than plain float2 loads.)
template <int PL>
struct LinkSh;
template <>
struct LinkSh<P64> {
    static constexpr int kBytes = 576;
    static __device__ __forceinline__ void pack(unsigned char* L, int T, int t, const char* U, long long V,
                                                long long s) {
        const double2* Ug = reinterpret_cast<const double2*>(U);
        double2* A = reinterpret_cast<double2*>(L);
        for (int c = 0; c < 36; ++c) A[c * T + t] = Ug[(long long)c * V + s];
    }
    template <class C>
    static __device__ __forceinline__ void load(const unsigned char* L, int T, int mu, int t, cx<C> u[9]) {
        const double2* A = reinterpret_cast<const double2*>(L) + mu * 9 * T;
#pragma unroll
        for (int c = 0; c < 9; ++c) {
            const double2 v = A[c * T + t];
            u[c] = mk<C>((C)v.x, (C)v.y);
        }
    }
};
template <>
struct LinkSh<P32> {
    static constexpr int kBytes = 288;
    static __device__ __forceinline__ void pack(unsigned char* L, int T, int t, const char* U, long long V,
                                                long long s) {
        const float2* Ug = reinterpret_cast<const float2*>(U);
        float2* A = reinterpret_cast<float2*>(L);
        for (int c = 0; c < 36; ++c) A[c * T + t] = Ug[(long long)c * V + s];
    }
    template <class C>
    static __device__ __forceinline__ void load(const unsigned char* L, int T, int mu, int t, cx<C> u[9]) {
        const float2* A = reinterpret_cast<const float2*>(L) + mu * 9 * T;
#pragma unroll
        for (int c = 0; c < 9; ++c) {
            const float2 v = A[c * T + t];
            u[c] = mk<C>((C)v.x, (C)v.y);
        }
    }
};
template <int PL>
struct LinkSh16 {
    static constexpr int kBytes = 144;
    static __device__ __forceinline__ void pack(unsigned char* L, int T, int t, const char* U, long long V,
                                                long long s) {
        const uint32_t* Ug = reinterpret_cast<const uint32_t*>(U);
        uint32_t* A = reinterpret_cast<uint32_t*>(L);            // uint4 [4][2][T] seen as words
        uint32_t* B = reinterpret_cast<uint32_t*>(L + 128 * T);  // uint32 [4][T]
        for (int mu = 0; mu < 4; ++mu) {
            for (int c = 0; c < 8; ++c)
                A[4 * ((mu * 2 + (c >> 2)) * T + t) + (c & 3)] = Ug[(long long)(mu * 9 + c) * V + s];
            B[mu * T + t] = Ug[(long long)(mu * 9 + 8) * V + s];
        }
    }
    template <class C>
    static __device__ __forceinline__ void load(const unsigned char* L, int T, int mu, int t, cx<C> u[9]) {
        constexpr int bf = (PL == PB16);
        const uint4* A = reinterpret_cast<const uint4*>(L) + mu * 2 * T;
        const uint32_t* B = reinterpret_cast<const uint32_t*>(L + 128 * T);
#pragma unroll
        for (int q = 0; q < 2; ++q) {
            const uint4 v = A[q * T + t];
            const float2 a = h2_to_f2(v.x, bf), b = h2_to_f2(v.y, bf), c = h2_to_f2(v.z, bf), d = h2_to_f2(v.w, bf);
            u[4 * q] = mk<C>((C)a.x, (C)a.y);
            u[4 * q + 1] = mk<C>((C)b.x, (C)b.y);
            u[4 * q + 2] = mk<C>((C)c.x, (C)c.y);
            u[4 * q + 3] = mk<C>((C)d.x, (C)d.y);
        }
        const float2 w = h2_to_f2(B[mu * T + t], bf);
        u[8] = mk<C>((C)w.x, (C)w.y);
    }
};
template <>
struct LinkSh<P16> : LinkSh16<P16> {};
template <>
struct LinkSh<PB16> : LinkSh16<PB16> {};

// The MR iterate rho in shared memory: FP32 as float4 [6][T] (two complex per
// load), FP64 as double2 [12][T].
template <class C>
__device__ __forceinline__ void rho_store(unsigned char* R, int T, int t, const cx<C> v[12]) {
    if constexpr (sizeof(C) == 4) {
        float4* p = reinterpret_cast<float4*>(R);
#pragma unroll
        for (int q = 0; q < 6; ++q) p[q * T + t] = make_float4(v[2 * q].re, v[2 * q].im, v[2 * q + 1].re, v[2 * q + 1].im);
    } else {
        double2* p = reinterpret_cast<double2*>(R);
#pragma unroll
        for (int c = 0; c < 12; ++c) p[c * T + t] = make_double2(v[c].re, v[c].im);
    }
}
template <class C>
__device__ __forceinline__ void rho_load(const unsigned char* R, int T, int t, cx<C> v[12]) {
    if constexpr (sizeof(C) == 4) {
        const float4* p = reinterpret_cast<const float4*>(R);
#pragma unroll
        for (int q = 0; q < 6; ++q) {
            const float4 a = p[q * T + t];
            v[2 * q] = mk<C>(a.x, a.y);
            v[2 * q + 1] = mk<C>(a.z, a.w);
        }
    } else {
        const double2* p = reinterpret_cast<const double2*>(R);
#pragma unroll
        for (int c = 0; c < 12; ++c) {
            const double2 a = p[c * T + t];
            v[c] = mk<C>(a.x, a.y);
        }
    }
}

template <class C>
__device__ __forceinline__ void block_sum3(C& a, C& b, C& c, C* red) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        a += __shfl_xor_sync(0xffffffffu, a, o);
        b += __shfl_xor_sync(0xffffffffu, b, o);
        c += __shfl_xor_sync(0xffffffffu, c, o);
    }
    const int w = threadIdx.x >> 5;
    if ((threadIdx.x & 31) == 0) {
        red[3 * w] = a;
        red[3 * w + 1] = b;
        red[3 * w + 2] = c;
    }
    __syncthreads();
    const int nw = blockDim.x >> 5;
    C sa = 0, sb = 0, sc = 0;
    for (int i = 0; i < nw; ++i) {
        sa += red[3 * i];
        sb += red[3 * i + 1];
        sc += red[3 * i + 2];
    }
    a = sa;
    b = sb;
    c = sc;
}

__device__ __forceinline__ unsigned smem_u32(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }
__device__ __forceinline__ unsigned long long global_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}
// mbarrier completed by the byte count of one bulk copy (one arrival)
__device__ __forceinline__ void bulk_copy_start(void* dst, const void* src, unsigned bytes, unsigned long long* bar) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(bar)) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
                 : "memory");
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                     smem_u32(dst)),
                 "l"(src), "r"(bytes), "r"(smem_u32(bar))
                 : "memory");
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
