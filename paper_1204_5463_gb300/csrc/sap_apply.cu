// The SAP preconditioner z = M v (Sec. 2, Algorithm 2; Sec. 4) with the domains'
// halos exchanged as half spinors.
//
// Every sweep takes, for each domain of its colour, r^l = (v - D x)^l, solves D^l y
// = r^l by MR steps and adds y to x^l. After its solve a domain sends one
// spin-projected half spinor of its new x, rounded as storage holds it, per face
// site and direction to the neighbouring domains' inboxes:
//   to the domain one step down in mu:  (1 + gamma_mu) x   (upper two rows; the
//       receiver owns the link and multiplies by U),
//   to the domain one step up in mu:    U^dagger (1 - gamma_mu) x.
// An inbox is contiguous, its slots in the order of a face's sites: the sites of a
// face read it through L2 in whole lines, half the bytes of a spinor and no link.
// The hops inside the domain come from the domain's own x in shared memory. x, in
// storage format, is all that is kept between sweeps. (The residual that the MR
// solve leaves could be carried along instead, with half spinors of y: a local
// stencil less a sweep, 298 us instead of 314 in the first line of the table below,
// 11.4 ms instead of 13.4 in its fourth. But the rounding of x then never enters r:
// FP32 errors of 1.8e-7 instead of 1.5e-7, and residuals of 4 u instead of 1.3 u
// after many cycles.)
//
// One CTA owns one domain (and right-hand side), one thread one site. Sweeps
// either run as one launch each, or, when the domains of one colour and all
// right-hand sides are resident together, as one cooperative launch with a
// barrier per right-hand side between sweeps: the CTA then fetches the links
// of its next domain while the barrier completes.
//
// What it replaces and what bounds it: sap_sweep_kernel reads the spinors and links
// of the halo from L2 one hop at a time (5.3 us of a 22 us sweep), and a launch per
// sweep costs 8-9 us between the sweeps of 256 domains. Its results are the
// same to the bit (in FP64 up to rounding). Calls, conversions included (5 cycles x 4 MR steps unless stated):
//   16^3 x 32, 4^4 domains, FP32                 343 -> 314 us
//   the same with the clover term (8 x 5)        759 -> 719 us
//   12^3 x 18, 3^4 domains, 3 BF16 rhs (4 x 5)   342 -> 284 us
//   24^3 x 48, 4^4 domains, 12 FP16 rhs         14.93 -> 13.38 ms
//   8^3 x 16, 2 rhs, solves on 4 streams         38.2 -> 28.7 ms a burst
// Three quarters are the MR steps, bound by the latency of shared memory at the 16
// warps that 128 registers allow, with its pipe busy three quarters of the time;
// paired, scalar and mixed forms of the hop's FP32 arithmetic are within 2% of one
// another.
#include <cuda.h>

#include <algorithm>
#include <map>
#include <mutex>

#include "internal.h"
#include "sap_common.cuh"

namespace dwk {

namespace {

constexpr int kChain = 2;  // su3_mul as chains of scalar FMAs

template <class C>
struct SapArgs {
    Geom g;
    C diag;
    FieldRef v, x;
    const char* Uimg;             // links of every domain as the shared-memory image of LinkWarp
    const unsigned short* faces;  // [ns / 2]: lower-face site | mu << 10 of an inbox slot
    int ns;                       // inbox slots per domain (two per face site and direction)
    char* inbox;                  // per rhs: [domain] of Half<C> boxes
    long long inbox_rs;
    RhsCols jtab;
    int nrhs, nmr;
    int s0, s1, nsweeps;          // sweeps of this launch, sweeps of the application (2 per cycle)
    const char* clov;
    unsigned long long wait_ns;   // limit of a wait for the previous sweep
    unsigned* bar;                // [2 * DW_MAX_RHS]: barrier and exit counts per rhs (left at zero)
    int* err_host;
};

// Shared-memory layouts in pieces of a warp's 32 sites, so that every plane lies at a compile-time offset from one address: with planes of T
// sites each load had its own address arithmetic, a sixth of an MR step's
// instructions.
//
// The site vectors x and rho: FP32 float4 [warp][6][32], FP64 double2 [warp][12][32].
template <class C>
struct SiteVec {
    static constexpr int kPlanes = sizeof(C) == 4 ? 6 : 12;
    static constexpr int kWarp = kPlanes * 512;  // bytes of 32 sites
    static __device__ __forceinline__ int at(int t) { return (t >> 5) * kWarp + (t & 31) * 16; }
    static __device__ __forceinline__ void store(unsigned char* p, const cx<C> v[12]) {
#pragma unroll
        for (int q = 0; q < kPlanes; ++q)
            if constexpr (sizeof(C) == 4)
                *reinterpret_cast<float4*>(p + 512 * q) =
                    make_float4(v[2 * q].re, v[2 * q].im, v[2 * q + 1].re, v[2 * q + 1].im);
            else
                *reinterpret_cast<double2*>(p + 512 * q) = make_double2(v[q].re, v[q].im);
    }
    static __device__ __forceinline__ void load(const unsigned char* p, cx<C> v[12]) {
#pragma unroll
        for (int q = 0; q < kPlanes; ++q)
            if constexpr (sizeof(C) == 4) {
                const float4 a = *reinterpret_cast<const float4*>(p + 512 * q);
                v[2 * q] = mk<C>(a.x, a.y);
                v[2 * q + 1] = mk<C>(a.z, a.w);
            } else {
                const double2 a = *reinterpret_cast<const double2*>(p + 512 * q);
                v[q] = mk<C>(a.x, a.y);
            }
    }
};

// The links of a domain, per warp [4 directions] of
//   P64      double2 [9][32]
//   P32      float4 [4][32] (entries 2q, 2q + 1), float2 [32] (entry 8)
//   P16/B16  uint4 [2][32] (entries 4q .. 4q + 3), uint32 [32] (entry 8)
template <int PL>
struct LinkWarp {
    static constexpr int kEntry = PL == P64 ? 16 : PL == P32 ? 8 : 4;  // bytes of one complex entry
    static constexpr int kMu = 9 * 32 * kEntry;                        // bytes of 32 sites' links in one direction
    static constexpr int kWarp = 4 * kMu;
    template <class C>
    static __device__ __forceinline__ void load(const unsigned char* L, int mu, int t, cx<C> u[9]) {
        const unsigned char* b = L + (t >> 5) * kWarp + mu * kMu;
        const unsigned char* p = b + (t & 31) * 16;
        if constexpr (PL == P64) {
#pragma unroll
            for (int c = 0; c < 9; ++c) {
                const double2 v = *reinterpret_cast<const double2*>(p + 512 * c);
                u[c] = mk<C>((C)v.x, (C)v.y);
            }
        } else if constexpr (PL == P32) {
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const float4 v = *reinterpret_cast<const float4*>(p + 512 * q);
                u[2 * q] = mk<C>((C)v.x, (C)v.y);
                u[2 * q + 1] = mk<C>((C)v.z, (C)v.w);
            }
            const float2 v = *reinterpret_cast<const float2*>(b + 2048 + (t & 31) * 8);
            u[8] = mk<C>((C)v.x, (C)v.y);
        } else {
            constexpr int bf = (PL == PB16);
#pragma unroll
            for (int q = 0; q < 2; ++q) {
                const uint4 v = *reinterpret_cast<const uint4*>(p + 512 * q);
                const float2 f0 = h2_to_f2(v.x, bf), f1 = h2_to_f2(v.y, bf), f2 = h2_to_f2(v.z, bf), f3 = h2_to_f2(v.w, bf);
                u[4 * q] = mk<C>((C)f0.x, (C)f0.y);
                u[4 * q + 1] = mk<C>((C)f1.x, (C)f1.y);
                u[4 * q + 2] = mk<C>((C)f2.x, (C)f2.y);
                u[4 * q + 3] = mk<C>((C)f3.x, (C)f3.y);
            }
            const float2 w = h2_to_f2(*reinterpret_cast<const uint32_t*>(b + 1024 + (t & 31) * 4), bf);
            u[8] = mk<C>((C)w.x, (C)w.y);
        }
    }
    static __device__ __forceinline__ void pack(unsigned char* L, int t, const char* U, long long V, long long s) {
        constexpr int N = PL == P64 ? 1 : PL == P32 ? 2 : 4;  // entries of a 16-byte word
        for (int mu = 0; mu < 4; ++mu)
            for (int c = 0; c < 9; ++c) {
                unsigned char* b = L + (t >> 5) * kWarp + mu * kMu + (c / N) * 512;
                unsigned char* to = (PL == P64 || c < 8) ? b + (t & 31) * 16 + (c % N) * kEntry : b + (t & 31) * kEntry;
                const long long e = (long long)(mu * 9 + c) * V + s;
                if constexpr (PL == P64)
                    *reinterpret_cast<double2*>(to) = reinterpret_cast<const double2*>(U)[e];
                else if constexpr (PL == P32)
                    *reinterpret_cast<float2*>(to) = reinterpret_cast<const float2*>(U)[e];
                else
                    *reinterpret_cast<uint32_t*>(to) = reinterpret_cast<const uint32_t*>(U)[e];
            }
    }
};

// Half spinors (the upper two spin rows) of an inbox in global memory, in boxes of 8
// slots: 16-byte words [3 or 6][8], read through L2 (other SMs write them)
template <class C>
struct Half {
    static constexpr int kWords = sizeof(C) == 4 ? 3 : 6;
    static constexpr int kBox = kWords * 128;
    static __host__ __device__ int bytes(int ns) { return (ns + 7) / 8 * kBox; }
    static __device__ __forceinline__ int at(int q) { return (q >> 3) * kBox + (q & 7) * 16; }
    static __device__ __forceinline__ void load(const unsigned char* p, cx<C> h0[3], cx<C> h1[3]) {
        if constexpr (sizeof(C) == 4) {
            const float4* w = reinterpret_cast<const float4*>(p);
            const float4 a = __ldcg(w), b = __ldcg(w + 8), c = __ldcg(w + 16);
            h0[0] = mk<C>(a.x, a.y), h0[1] = mk<C>(a.z, a.w), h0[2] = mk<C>(b.x, b.y);
            h1[0] = mk<C>(b.z, b.w), h1[1] = mk<C>(c.x, c.y), h1[2] = mk<C>(c.z, c.w);
        } else {
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                const double2* w = reinterpret_cast<const double2*>(p) + 8 * i;
                const double2 a = __ldcg(w), b = __ldcg(w + 24);
                h0[i] = mk<C>(a.x, a.y);
                h1[i] = mk<C>(b.x, b.y);
            }
        }
    }
    static __device__ __forceinline__ void store(unsigned char* p, const cx<C> h0[3], const cx<C> h1[3]) {
        if constexpr (sizeof(C) == 4) {
            *reinterpret_cast<float4*>(p) = make_float4(h0[0].re, h0[0].im, h0[1].re, h0[1].im);
            *reinterpret_cast<float4*>(p + 128) = make_float4(h0[2].re, h0[2].im, h1[0].re, h1[0].im);
            *reinterpret_cast<float4*>(p + 256) = make_float4(h1[1].re, h1[1].im, h1[2].re, h1[2].im);
        } else {
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                *reinterpret_cast<double2*>(p + 128 * i) = make_double2(h0[i].re, h0[i].im);
                *reinterpret_cast<double2*>(p + 128 * (3 + i)) = make_double2(h1[i].re, h1[i].im);
            }
        }
    }
};

// what a face site sends: SIDE 0, its lower face: (1 + gamma_MU) x; SIDE 1,
// its upper face: U^dagger (1 - gamma_MU) x
template <int MU, class C, class LW>
__device__ __forceinline__ void face_half(int side, const cx<C> x[12], const unsigned char* lsh, int t, cx<C> k0[3],
                                          cx<C> k1[3]) {
    if (side == 0) {
        project<MU, +1, C>(x, k0, k1);
    } else {
        cx<C> h0[3], h1[3], u[9];
        project<MU, -1, C>(x, h0, h1);
        LW::template load<C>(lsh, MU, t, u);
        su3_mul<C, true, kChain>(u, h0, k0);
        su3_mul<C, true, kChain>(u, h1, k1);
    }
}

// acc += m times the spin rows rebuilt from k0, k1 (m = 0: a neighbour outside the domain)
template <int MU, int SIGN, class C>
__device__ __forceinline__ void reconstruct_if(C m, const cx<C> k0[3], const cx<C> k1[3], cx<C> acc[12]) {
    const C s = SIGN > 0 ? m : -m;
    auto add = [](cx<C>& to, C w, cx<C> k) { to = mk<C>(fma(w, k.re, to.re), fma(w, k.im, to.im)); };
    auto addi = [](cx<C>& to, C w, cx<C> k) { to = mk<C>(fma(-w, k.im, to.re), fma(w, k.re, to.im)); };  // + i w k
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        add(acc[c], m, k0[c]);
        add(acc[3 + c], m, k1[c]);
        if constexpr (MU == 0) {
            addi(acc[6 + c], s, k1[c]);
            addi(acc[9 + c], s, k0[c]);
        } else if constexpr (MU == 1) {
            add(acc[6 + c], s, k1[c]);
            add(acc[9 + c], -s, k0[c]);
        } else if constexpr (MU == 2) {
            addi(acc[6 + c], s, k0[c]);
            addi(acc[9 + c], -s, k1[c]);
        } else {
            add(acc[6 + c], s, k0[c]);
            add(acc[9 + c], s, k1[c]);
        }
    }
}
template <int MU, int SIGN, class C>
__device__ __forceinline__ void hop_if(bool in, const cx<C> psi[12], const cx<C> u[9], cx<C> acc[12]) {
    cx<C> h0[3], h1[3], k0[3], k1[3];
    project<MU, SIGN, C>(psi, h0, h1);
    su3_mul<C, (SIGN < 0), kChain>(u, h0, k0);
    su3_mul<C, (SIGN < 0), kChain>(u, h1, k1);
    reconstruct_if<MU, SIGN, C>(in ? C(1) : C(0), k0, k1, acc);
}

// CTA-wide sums of three numbers, at most 8 warps: within a warp the three
// are folded together (lanes end up with one number each), then every thread adds
// the warps' sums in order. red: [8][4].
template <class C>
__device__ __forceinline__ void cta_sum3(C& a, C& b, C& c, C* red) {
    constexpr unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31, nw = blockDim.x >> 5;
    const bool h16 = lane & 16, h8 = lane & 8;
    // lanes 0-15 keep (a, b), lanes 16-31 (c, 0); then groups of 8 lanes a, b, c, 0
    const C k0 = (h16 ? c : a) + __shfl_xor_sync(full, h16 ? a : c, 16);
    const C k1 = (h16 ? C(0) : b) + __shfl_xor_sync(full, h16 ? b : C(0), 16);
    C k = (h8 ? k1 : k0) + __shfl_xor_sync(full, h8 ? k0 : k1, 8);
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) k += __shfl_xor_sync(full, k, o);
    if ((lane & 7) == 0) red[4 * (threadIdx.x >> 5) + (lane >> 3)] = k;
    __syncthreads();
    a = b = c = C(0);
    for (int w = 0; w < nw; ++w) {
        a += red[4 * w];
        b += red[4 * w + 1];
        c += red[4 * w + 2];
    }
}

// waits until *cnt reaches target, giving up after limit ns
__device__ __forceinline__ bool count_wait(const unsigned* cnt, unsigned target, unsigned long long limit) {
    const unsigned long long t0 = global_ns();
    for (unsigned it = 1;; ++it) {
        unsigned v;
        asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(cnt) : "memory");
        if (v >= target) return true;
        if ((it & 255) == 0 && global_ns() - t0 > limit) return false;
    }
}

template <int PS, int PL, class C, bool CLOV>
__global__ void __launch_bounds__(256, sizeof(C) == 4 ? 2 : 1) sap_apply_kernel(const __grid_constant__ SapArgs<C> a) {
    constexpr int CP = (sizeof(C) == 4) ? P32 : P64;  // storage of the clover term
    typedef LinkWarp<PL> LW;
    typedef SiteVec<C> SV;
    typedef Half<C> HB;
    extern __shared__ __align__(16) unsigned char smem[];
    const Geom& g = a.g;
    const int T = blockDim.x, ns = a.ns, hbytes = HB::bytes(ns);
    unsigned char* rsh = smem;                                  // x, then rho, then the new x
    unsigned char* lsh = smem + SV::kWarp * (T >> 5);           // links
    C* red = reinterpret_cast<C*>(lsh + LW::kWarp * (T >> 5));  // [8][4]
    unsigned long long* lbar = reinterpret_cast<unsigned long long*>(red + 32);

    const int r = blockIdx.x % a.nrhs;
    const int e = blockIdx.x / a.nrhs;
    if (!rhs_active(a.jtab, r)) return;  // every CTA of this rhs
    const char* vb = field_ptr(a.v, a.jtab, r);
    char* xb = field_ptr(a.x, a.jtab, r);
    unsigned char* inb = reinterpret_cast<unsigned char*>(a.inbox) + (long long)r * a.inbox_rs;
    const unsigned ncta = (unsigned)g.ndom / 2;  // CTAs of this rhs

    const int tid = threadIdx.x;
    const bool act = tid < g.B;
    int lx[4];
    {
        int q = act ? tid : 0;
        lx[0] = q % g.b[0];
        q /= g.b[0];
        lx[1] = q % g.b[1];
        q /= g.b[1];
        lx[2] = q % g.b[2];
        lx[3] = q / g.b[2];
    }
    const int ls1 = g.b[0], ls2 = g.b[0] * g.b[1], ls3 = g.b[0] * g.b[1] * g.b[2];  // in-domain strides
    const unsigned lbytes = (unsigned)LW::kWarp * (unsigned)(T >> 5);
    unsigned char* own = rsh + SV::at(tid);
    const unsigned char* limg = reinterpret_cast<const unsigned char*>(a.Uimg);
    const int dst1 = g.nb[0], dst2 = dst1 * g.nb[1], dst3 = dst2 * g.nb[2];

    int D[4], dom;
    // domain e of a colour: block coordinates D with sum(D) % 2 == colour
    auto locate = [&](int colour) {
        const int half1 = g.nb[0] >> 1;
        int t = e / half1;
        D[1] = t % g.nb[1];
        t /= g.nb[1];
        D[2] = t % g.nb[2];
        D[3] = t / g.nb[2];
        D[0] = 2 * (e % half1) + ((colour + D[1] + D[2] + D[3]) & 1);
        dom = D[0] + dst1 * D[1] + dst2 * D[2] + dst3 * D[3];
    };
    auto links_start = [&]() {
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(lbar)), "r"(lbytes)
                     : "memory");
        asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                         smem_u32(lsh)),
                     "l"(limg + (long long)dom * lbytes), "r"(lbytes), "r"(smem_u32(lbar))
                     : "memory");
    };
    // programmatic dependent launch: the next sweep's CTAs may be scheduled as
    // this one's retire, and stage their links meanwhile
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    locate(a.s0 & 1);
    if (tid == 0) {
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(lbar)) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        links_start();
    }
    // everything but the links depends on the previous kernel of the stream
    asm volatile("griddepcontrol.wait;" ::: "memory");
    __syncthreads();  // the mbarrier is initialised before any thread waits on it

    const C diag2 = 2 * a.diag;
    // inbox slots of this site's lines in the four directions
    const int q0 = lx[1] + g.b[1] * (lx[2] + g.b[2] * lx[3]);
    const int q1 = g.B / g.b[0] + lx[0] + g.b[0] * (lx[2] + g.b[2] * lx[3]);
    const int q2 = g.B / g.b[0] + g.B / g.b[1] + lx[0] + g.b[0] * (lx[1] + g.b[1] * lx[3]);
    const int q3 = g.B / g.b[0] + g.B / g.b[1] + g.B / g.b[2] + lx[0] + g.b[0] * (lx[1] + g.b[1] * lx[2]);
    bool dead = false;
    for (int sw = a.s0; sw < a.s1; ++sw) {
        const bool first = sw < 2;  // x^l is still zero
        long long s;
        {
            int xg[4];
            xg[0] = D[0] * g.b[0] + lx[0];
            xg[1] = D[1] * g.b[1] + lx[1];
            xg[2] = D[2] * g.b[2] + lx[2];
            xg[3] = D[3] * g.b[3] + lx[3];
            s = site_index(g, xg);
        }
        cx<C> rho[12], y[12];
        // the domain's own iterate (written by this thread two sweeps ago) and v
        if (act) {
            if (!first) {
                load_spinor<PS, C, 2>(xb, g.V, s, y);
                SV::store(own, y);
            }
            if (sw == 0) load_spinor<PS, C>(vb, g.V, s, rho);
        } else {
#pragma unroll
            for (int c = 0; c < 12; ++c) rho[c] = czero<C>();
        }
        // the previous sweep's sends have arrived
        bool ok = true;
        if (sw > a.s0) {
            if (tid == 0) ok = count_wait(a.bar + r, ncta * (unsigned)(sw - a.s0), a.wait_ns);
            __syncthreads();
        }
        ok = ok && bulk_copy_wait(lbar, (sw - a.s0) & 1);
        if (__syncthreads_or(!ok)) {
            if (tid == 0) {
                *reinterpret_cast<volatile int*>(a.err_host) = 1;
                __threadfence_system();
            }
            bulk_copy_wait(lbar, (sw - a.s0) & 1);  // the copy may still be in flight: wait before the CTA retires
            dead = true;
            break;
        }
        // r = v - D x at this site: neighbours inside the domain from shared memory,
        // the others' half spinors from the inbox (fetched one direction ahead)
        if (act && sw > 0) {
            cx<C> acc[12], e0[3], e1[3];
#pragma unroll
            for (int c = 0; c < 12; ++c) acc[c] = czero<C>();
            const unsigned char* box = inb + (long long)dom * hbytes;
#define SAP_FETCH(MU)                                                                        \
    {                                                                                        \
        if (lx[MU] + 1 == g.b[MU])                                                           \
            HB::load(box + HB::at(q##MU), e0, e1);                                           \
        else if (lx[MU] == 0)                                                                \
            HB::load(box + HB::at(ns / 2 + q##MU), e0, e1);                                  \
    }
#define SAP_RES_HOPS(MU, LS_MU, NEXT)                                                        \
    {                                                                                        \
        const bool up = lx[MU] + 1 < g.b[MU], dn = lx[MU] >= 1;                              \
        cx<C> psi[12], u[9], h0[3], h1[3], k0[3], k1[3], f0[3], f1[3];                       \
        _Pragma("unroll") for (int c = 0; c < 3; ++c) f0[c] = e0[c], f1[c] = e1[c];          \
        NEXT;                                                                                \
        SV::load(rsh + SV::at(up ? tid + LS_MU : tid), psi);                                 \
        project<MU, +1, C>(psi, h0, h1);                                                     \
        _Pragma("unroll") for (int c = 0; c < 3; ++c) {                                      \
            h0[c] = up ? h0[c] : f0[c];                                                      \
            h1[c] = up ? h1[c] : f1[c];                                                      \
        }                                                                                    \
        LW::template load<C>(lsh, MU, tid, u);                                               \
        su3_mul<C, false, kChain>(u, h0, k0);                                                \
        su3_mul<C, false, kChain>(u, h1, k1);                                                \
        reconstruct<MU, +1, C>(k0, k1, acc);                                                 \
        if (!up && !dn) HB::load(box + HB::at(ns / 2 + q##MU), f0, f1);                      \
        const int td = dn ? tid - LS_MU : tid;                                               \
        SV::load(rsh + SV::at(td), psi);                                                     \
        LW::template load<C>(lsh, MU, td, u);                                                \
        project<MU, -1, C>(psi, h0, h1);                                                     \
        su3_mul<C, true, kChain>(u, h0, k0);                                                 \
        su3_mul<C, true, kChain>(u, h1, k1);                                                 \
        _Pragma("unroll") for (int c = 0; c < 3; ++c) {                                      \
            k0[c] = dn ? k0[c] : f0[c];                                                      \
            k1[c] = dn ? k1[c] : f1[c];                                                      \
        }                                                                                    \
        reconstruct<MU, -1, C>(k0, k1, acc);                                                 \
    }
#define SAP_IN_HOPS(MU)                                                                      \
    {                                                                                        \
        cx<C> u[9], h0[3], h1[3], k0[3], k1[3];                                              \
        if (lx[MU] + 1 == g.b[MU]) {                                                         \
            HB::load(box + HB::at(q##MU), h0, h1);                                           \
            LW::template load<C>(lsh, MU, tid, u);                                           \
            su3_mul<C, false, kChain>(u, h0, k0);                                            \
            su3_mul<C, false, kChain>(u, h1, k1);                                            \
            reconstruct<MU, +1, C>(k0, k1, acc);                                             \
        }                                                                                    \
        if (lx[MU] == 0) {                                                                   \
            HB::load(box + HB::at(ns / 2 + q##MU), k0, k1);                                  \
            reconstruct<MU, -1, C>(k0, k1, acc);                                             \
        }                                                                                    \
    }
            if (first) {
                SAP_IN_HOPS(0)
                SAP_IN_HOPS(1)
                SAP_IN_HOPS(2)
                SAP_IN_HOPS(3)
                load_spinor<PS, C>(vb, g.V, s, rho);
            } else {
                SAP_FETCH(0)
                SAP_RES_HOPS(0, 1, SAP_FETCH(1))
                SAP_RES_HOPS(1, ls1, SAP_FETCH(2))
                SAP_RES_HOPS(2, ls2, SAP_FETCH(3))
                load_spinor<PS, C>(vb, g.V, s, rho);
                SAP_RES_HOPS(3, ls3, )
            }
#undef SAP_RES_HOPS
#undef SAP_IN_HOPS
#undef SAP_FETCH
            const C half = (C)0.5;
            if (first) {
#pragma unroll
                for (int c = 0; c < 12; ++c) rho[c] = rho[c] + half * acc[c];
            } else {
                SV::load(own, y);
                if constexpr (CLOV) clover_acc<CP, C>(a.clov, g.V, s, y, acc, (C)-2);  // A x as -2 A x in acc
#pragma unroll
                for (int c = 0; c < 12; ++c) rho[c] = rho[c] - (a.diag * y[c] - half * acc[c]);
            }
        }
        if (!first) __syncthreads();  // x makes room for the MR iterate
#pragma unroll
        for (int c = 0; c < 12; ++c) y[c] = czero<C>();

        // MR on D^l y = r^l out of shared memory, with p = 2 D^l rho:
        // beta = <p, rho> / <p, p>, y += 2 beta rho, rho -= beta p
        for (int it = 0; it < a.nmr; ++it) {
            cx<C> p[12];  // the hops, then p
            SV::store(own, rho);
#pragma unroll
            for (int c = 0; c < 12; ++c) p[c] = czero<C>();
            __syncthreads();
            C pr_re = 0, pr_im = 0, pp = 0;
            if (act) {
                cx<C> psi[12], u[9];
                // directions 0 to 2 without branches, so that the loads of one hop
                // overlap the arithmetic of another (a neighbour outside the domain
                // is the site itself, with weight 0); direction 3, whose hops whole
                // warps skip at the domain's ends, with them
#define SAP_ALL_HOPS(MU, LS_MU)                          \
    {                                                    \
        const bool up = lx[MU] + 1 < g.b[MU], dn = lx[MU] >= 1; \
        const int tu = up ? tid + LS_MU : tid, td = dn ? tid - LS_MU : tid; \
        SV::load(rsh + SV::at(tu), psi);                 \
        LW::template load<C>(lsh, MU, tid, u);           \
        hop_if<MU, +1, C>(up, psi, u, p);                \
        SV::load(rsh + SV::at(td), psi);                 \
        LW::template load<C>(lsh, MU, td, u);            \
        hop_if<MU, -1, C>(dn, psi, u, p);                \
    }
                SAP_ALL_HOPS(0, 1)
                SAP_ALL_HOPS(1, ls1)
                SAP_ALL_HOPS(2, ls2)
#undef SAP_ALL_HOPS
                if (lx[3] + 1 < g.b[3]) {
                    SV::load(rsh + SV::at(tid + ls3), psi);
                    LW::template load<C>(lsh, 3, tid, u);
                    hop<3, +1, C, kChain>(psi, u, p);
                }
                if (lx[3] >= 1) {
                    SV::load(rsh + SV::at(tid - ls3), psi);
                    LW::template load<C>(lsh, 3, tid - ls3, u);
                    hop<3, -1, C, kChain>(psi, u, p);
                }
                // the site's own rho is read back from shared memory (where the
                // neighbours read it) rather than kept in registers over the hops:
                // the 24 registers go to overlapping the hops' loads
                SV::load(own, rho);
                if constexpr (CLOV) clover_acc<CP, C>(a.clov, g.V, s, rho, p, (C)-2);  // A rho as -2 A rho
#pragma unroll
                for (int c = 0; c < 12; ++c) {
                    p[c] = mk<C>(fma(diag2, rho[c].re, -p[c].re), fma(diag2, rho[c].im, -p[c].im));
                    const cx<C> t = cmulc(p[c], rho[c]);
                    pr_re += t.re;
                    pr_im += t.im;
                    pp += p[c].re * p[c].re + p[c].im * p[c].im;
                }
            }
            cta_sum3(pr_re, pr_im, pp, red);
            if (pp > (C)0) {
                const cx<C> beta = mk<C>(pr_re / pp, pr_im / pp), alpha = beta + beta;
#pragma unroll
                for (int c = 0; c < 12; ++c) {
                    y[c] = y[c] + alpha * rho[c];
                    rho[c] = rho[c] - beta * p[c];
                }
            }
        }

        // x^l <- x^l + y^l
        if (act && !first) {
            cx<C> xo[12];
            load_spinor<PS, C, 2>(xb, g.V, s, xo);
#pragma unroll
            for (int c = 0; c < 12; ++c) y[c] = y[c] + xo[c];
        }
        // the half spinors of x, as storage holds it, to the neighbouring domains' inboxes
        if (sw + 1 < a.nsweeps) {
            {
                cx<C> kept[12];
#pragma unroll
                for (int c = 0; c < 12; ++c) kept[c] = y[c];
                round_spinor<PS, C>(kept);
                SV::store(own, kept);
            }
            __syncthreads();
            for (int q = tid; q < ns; q += T) {
                const int side = q >= ns / 2 ? 1 : 0;
                const int f = __ldg(a.faces + q - side * (ns / 2)), mu = f >> 10;
                int t = f & 1023;
                cx<C> xx[12], k0[3], k1[3];
                long long to;
#define SAP_SEND(MU, LS_MU, DST)                                                             \
    {                                                                                        \
        if (side) {                                                                          \
            t += (g.b[MU] - 1) * LS_MU;                                                      \
            to = D[MU] + 1 < g.nb[MU] ? dom + DST : dom - (g.nb[MU] - 1) * DST;              \
        } else {                                                                             \
            to = D[MU] > 0 ? dom - DST : dom + (g.nb[MU] - 1) * DST;                         \
        }                                                                                    \
        SV::load(rsh + SV::at(t), xx);                                                       \
        face_half<MU, C, LW>(side, xx, lsh, t, k0, k1);                                      \
    }
                if (mu == 0)
                    SAP_SEND(0, 1, 1)
                else if (mu == 1)
                    SAP_SEND(1, ls1, dst1)
                else if (mu == 2)
                    SAP_SEND(2, ls2, dst2)
                else
                    SAP_SEND(3, ls3, dst3)
#undef SAP_SEND
                HB::store(inb + to * hbytes + HB::at(q), k0, k1);
            }
        }
        const long long sc = s;  // this sweep's site
        if (sw + 1 < a.s1) {
            __syncthreads();  // all sends are issued, and nobody reads this domain's links any more
            locate((sw + 1) & 1);
            if (tid == 0) {
                asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(a.bar + r) : "memory");
                links_start();
            }
        }
        if (act) store_spinor<PS, C>(xb, g.V, sc, y);
    }
    // the last CTA of this rhs leaves the counters at zero for the next launch
    if (!dead && a.s1 - a.s0 > 1 && tid == 0) {
        unsigned* ex = a.bar + DW_MAX_RHS + r;
        if (atomicAdd(ex, 1u) == ncta - 1) {
            a.bar[r] = 0u;
            *ex = 0u;
        }
    }
}

// The links of domain blockIdx.x (both colours) as LinkWarp keeps them in shared
// memory. Block 0 also writes what follows the image: faces[q], the lower-face site |
// mu << 10 of inbox slot q (and of its mirror q + ns / 2), and the counters at zero.
template <int PL>
__global__ void warp_image_kernel(Geom g, const char* __restrict__ U, char* __restrict__ img, unsigned short* faces,
                                  unsigned* bar) {
    const int t = threadIdx.x;
    if (blockIdx.x == 0 && t < 2 * DW_MAX_RHS) bar[t] = 0u;
    if (t >= g.B) return;
    if (blockIdx.x == 0) {
        int ls = 1, off = 0;
        for (int mu = 0; mu < 4; ++mu) {
            if ((t / ls) % g.b[mu] == 0)  // the slots run over the other three coordinates in order
                faces[off + t % ls + ls * (t / (ls * g.b[mu]))] = (unsigned short)(t | (mu << 10));
            off += g.B / g.b[mu];
            ls *= g.b[mu];
        }
    }
    int D[4], q = blockIdx.x;
    D[0] = q % g.nb[0];
    q /= g.nb[0];
    D[1] = q % g.nb[1];
    q /= g.nb[1];
    D[2] = q % g.nb[2];
    D[3] = q / g.nb[2];
    int xg[4], r = t;
    for (int j = 0; j < 3; ++j) {
        xg[j] = D[j] * g.b[j] + r % g.b[j];
        r /= g.b[j];
    }
    xg[3] = D[3] * g.b[3] + r;
    LinkWarp<PL>::pack(reinterpret_cast<unsigned char*>(img) + (size_t)blockIdx.x * LinkWarp<PL>::kWarp * (blockDim.x >> 5),
                       t, U, g.V, site_index(g, xg));
}

// SMs that the stream's kernels may use: all, or those of its green context. The
// driver's functions are asked for by name (the library does not link libcuda);
// without them, the device's count.
int stream_sms(cudaStream_t st, int dev, int* sms) {
    typedef CUresult (*stream_ctx_t)(CUstream, CUcontext*);
    typedef CUresult (*ctx_resource_t)(CUcontext, CUdevResource*, CUdevResourceType);
    struct Driver {
        stream_ctx_t stream_ctx = nullptr;
        ctx_resource_t ctx_resource = nullptr;
        Driver() {
            void *a = nullptr, *b = nullptr;
            if (cudaGetDriverEntryPointByVersion("cuStreamGetCtx", &a, 12000, cudaEnableDefault) == cudaSuccess &&
                cudaGetDriverEntryPointByVersion("cuCtxGetDevResource", &b, 12040, cudaEnableDefault) == cudaSuccess) {
                stream_ctx = reinterpret_cast<stream_ctx_t>(a);
                ctx_resource = reinterpret_cast<ctx_resource_t>(b);
            }
            cudaGetLastError();
        }
    };
    static const Driver d;
    CUcontext ctx = nullptr;
    CUdevResource res;
    if (d.stream_ctx && d.ctx_resource && d.stream_ctx(reinterpret_cast<CUstream>(st), &ctx) == CUDA_SUCCESS &&
        d.ctx_resource(ctx, &res, CU_DEV_RESOURCE_TYPE_SM) == CUDA_SUCCESS) {
        *sms = (int)res.sm.smCount;
        return DW_OK;
    }
    DW_CUDA_TRY(cudaDeviceGetAttribute(sms, cudaDevAttrMultiProcessorCount, dev));
    return DW_OK;
}

template <int PS, int PL, class C>
int sap_apply_t(const Geom& g, double m0, FieldRef v, FieldRef x, const SapWork& w, RhsCols jtab, int nrhs,
                int ncycles, int nmr, cudaStream_t st, const ClovRef* cl, Profiler* prof, double bytes_first,
                double bytes_next) {
    const int threads = sap_threads(g);
    const size_t smem = (size_t)sap_apply_smem(PS, PL, g);
    const void* fn = cl ? (const void*)sap_apply_kernel<PS, PL, C, true> : (const void*)sap_apply_kernel<PS, PL, C, false>;
    // per device and CTA shape: the shared-memory limit is raised once, and the
    // CTAs that an SM holds at a time are asked for once
    static std::mutex mu;
    static std::map<std::pair<int, std::pair<const void*, std::pair<int, size_t>>>, int> resident;
    int dev = 0, fit = 0, sms = 0, rc;
    DW_CUDA_TRY(cudaGetDevice(&dev));
    if ((rc = stream_sms(st, dev, &sms))) return rc;
    {
        std::lock_guard<std::mutex> lock(mu);
        const auto key = std::make_pair(dev, std::make_pair(fn, std::make_pair(threads, smem)));
        auto it = resident.find(key);
        if (it == resident.end()) {
            int per = 0;
            DW_CUDA_TRY(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024));
            DW_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, fn, threads, smem));
            it = resident.emplace(key, per).first;
        }
        fit = sms * it->second;
    }
    SapArgs<C> a;
    a.g = g;
    a.diag = (C)(4.0 + m0);
    a.v = v;
    a.x = x;
    a.Uimg = w.Uimg;
    a.faces = sap_apply_faces(PL, g, w.Uimg);
    a.ns = sap_inbox_slots(g);
    a.inbox = w.inbox;
    a.inbox_rs = w.inbox_rs;
    a.jtab = jtab;
    a.nrhs = nrhs;
    a.nmr = nmr;
    a.nsweeps = 2 * ncycles;
    a.clov = cl ? ((sizeof(C) == 4) ? cl->a32 : cl->a64) : nullptr;
    // two seconds unless the context says otherwise, and more than an MR step takes in
    // any precision (70 us in FP64) for each of the steps by which another domain may be
    // behind
    a.wait_ns = w.wait_ns == SapWork::kWait ? w.wait_ns + 200000ULL * (unsigned long long)nmr : w.wait_ns;
    a.bar = sap_apply_counters(PL, g, w.Uimg);
    a.err_host = w.err;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(g.ndom / 2) * (unsigned)nrhs);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    void* args[] = {&a};
    int sw = 0;
    if ((long long)cfg.gridDim.x <= fit) {
        attr[0].id = cudaLaunchAttributeCooperative;
        attr[0].val.cooperative = 1;
        // at most 256 sweeps a launch: the barrier's counter stays small and no
        // launch holds the device for long, however many cycles are asked for
        for (; sw < a.nsweeps; sw = a.s1) {
            a.s0 = sw;
            a.s1 = std::min(a.nsweeps, sw + 256);
            const double bytes = (sw ? 0.0 : 2.0 * (bytes_first - bytes_next)) + (a.s1 - a.s0) * bytes_next;
            ProfScope ps(prof, "sap_sweep", bytes, a.s1 - a.s0);
            const cudaError_t e = cudaLaunchKernelExC(&cfg, fn, args);
            // refused for want of room: the remaining sweeps take a launch each
            if (e == cudaErrorCooperativeLaunchTooLarge || e == cudaErrorNotSupported) {
                cudaGetLastError();
                break;
            }
            DW_CUDA_TRY(e);
            DW_LAUNCH_CHECK();
        }
    }
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    for (; sw < a.nsweeps; ++sw) {
        a.s0 = sw;
        a.s1 = sw + 1;
        ProfScope ps(prof, "sap_sweep", sw < 2 ? bytes_first : bytes_next);
        DW_CUDA_TRY(cudaLaunchKernelExC(&cfg, fn, args));
        DW_LAUNCH_CHECK();
    }
    return DW_OK;
}

}  // namespace

int sap_inbox_slots(const Geom& g) {
    int n = 0;
    for (int j = 0; j < 4; ++j) n += 2 * (g.B / g.b[j]);
    return n;
}

int sap_apply_smem(int pspin, int plink, const Geom& g) {
    const int c = (pspin == P64) ? 8 : 4, T = sap_threads(g);
    return c * 24 * T + (int)(sap_link_image_bytes(plink, g) / g.ndom) + c * 32 + 16;
}

// Domains of at most 256 sites whose inbox is no larger than a double-precision
// field (the scratch that a solve has at hand).
bool sap_apply_fits(int prec, const Geom& g) {
    return g.B <= 256 && sap_inbox_bytes(prec, g) <= 192 * (size_t)g.V && sap_apply_smem(prec, prec, g) <= 227 * 1024;
}

size_t sap_inbox_bytes(int prec, const Geom& g) {
    const int ns = sap_inbox_slots(g);
    return (size_t)g.ndom * (prec == P64 ? Half<double>::bytes(ns) : Half<float>::bytes(ns));
}

size_t sap_apply_image_bytes(int prec, const Geom& g) {
    return sap_link_image_bytes(prec, g) + (sap_inbox_slots(g) / 2 * sizeof(unsigned short) + 15) / 16 * 16 +
           2 * DW_MAX_RHS * sizeof(unsigned);
}

unsigned short* sap_apply_faces(int prec, const Geom& g, char* img) {
    return reinterpret_cast<unsigned short*>(img + sap_link_image_bytes(prec, g));
}

unsigned* sap_apply_counters(int prec, const Geom& g, char* img) {
    return reinterpret_cast<unsigned*>(img + sap_apply_image_bytes(prec, g)) - 2 * DW_MAX_RHS;
}

int launch_sap_apply_image(int prec, const Geom& g, const char* U, char* img, cudaStream_t st) {
    const int T = sap_threads(g);
    static_assert(2 * DW_MAX_RHS <= 32, "a counter per thread of the smallest block");
    if (T != g.B) DW_CUDA_TRY(cudaMemsetAsync(img, 0, sap_link_image_bytes(prec, g), st));  // rows of idle threads
    const unsigned nb = (unsigned)g.ndom;
    unsigned short* faces = sap_apply_faces(prec, g, img);
    unsigned* bar = sap_apply_counters(prec, g, img);
    if (prec == P64)
        warp_image_kernel<P64><<<nb, T, 0, st>>>(g, U, img, faces, bar);
    else if (prec == P32)
        warp_image_kernel<P32><<<nb, T, 0, st>>>(g, U, img, faces, bar);
    else if (prec == P16)
        warp_image_kernel<P16><<<nb, T, 0, st>>>(g, U, img, faces, bar);
    else
        warp_image_kernel<PB16><<<nb, T, 0, st>>>(g, U, img, faces, bar);
    DW_LAUNCH_CHECK();
    return DW_OK;
}

int launch_sap_apply(int prec, const Geom& g, double m0, FieldRef v, FieldRef x, const SapWork& w, RhsCols jtab,
                     int nrhs, int ncycles, int nmr, cudaStream_t st, const ClovRef* cl, Profiler* prof,
                     double bytes_first, double bytes_next) {
    if (prec == P64)
        return sap_apply_t<P64, P64, double>(g, m0, v, x, w, jtab, nrhs, ncycles, nmr, st, cl, prof, bytes_first,
                                             bytes_next);
    if (prec == P32)
        return sap_apply_t<P32, P32, float>(g, m0, v, x, w, jtab, nrhs, ncycles, nmr, st, cl, prof, bytes_first,
                                            bytes_next);
    if (prec == P16)
        return sap_apply_t<P16, P16, float>(g, m0, v, x, w, jtab, nrhs, ncycles, nmr, st, cl, prof, bytes_first,
                                            bytes_next);
    if (prec == PB16)
        return sap_apply_t<PB16, PB16, float>(g, m0, v, x, w, jtab, nrhs, ncycles, nmr, st, cl, prof, bytes_first,
                                              bytes_next);
    return fail(DW_EINVAL, "unsupported SAP precision");
}

}  // namespace dwk
