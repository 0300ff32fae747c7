// The SAP preconditioner z = M v (Sec. 2, Algorithm 2; Sec. 4) with the residual
// carried along instead of recomputed.
//
// Algorithm 2 takes, for every domain it sweeps, r^l = (v - D x)^l. Between two
// visits of a domain only its neighbours' iterates change, so
//   r^l = rho^l + 1/2 sum over the hops that enter L^l of the neighbours' last
//         corrections y,
// where rho^l is the residual that the domain's own MR solve left. A domain
// therefore keeps rho^l, and after its solve sends one spin-projected half
// spinor per face site and direction to the neighbouring domains' inboxes:
//   to the domain one step down in mu:  (1 + gamma_mu) y   (upper two rows; the
//       receiver owns the link and multiplies by U),
//   to the domain one step up in mu:    U^dagger (1 - gamma_mu) y.
// An inbox is contiguous, so a domain fetches its whole halo with coalesced
// 16-byte copies and the residual costs only the hops that cross its faces.
//
// One CTA owns one domain (and right-hand side), one thread one site. Sweeps
// either run as one launch each, or, when the domains of one colour and all
// right-hand sides are resident together, as one cooperative launch with a
// barrier per right-hand side between sweeps: the CTA then fetches the links
// of its next domain while the barrier completes.
//
// What it replaces and what bounds it: recomputing r costs every sweep the full
// stencil (1392 flop a site), whose halo reads leave L2 one hop at a time
// (5.3 us of a 22 us sweep), and a launch per sweep costs 8-9 us between the
// sweeps of 256 domains. Here the residual takes 1.8 us, and the sends 1.2 us.
// Measured against one launch of sap_sweep_kernel per sweep (5 cycles x 4 MR
// steps unless stated): 8^3 x 16, 2 rhs served on 4 streams 37.4 -> 30.9 ms a
// burst; 12^3 x 18 in 3^4 domains, 3 BF16 rhs 343 -> 298 us; 24^3 x 48, 12 FP16
// rhs 14.92 -> 13.50 ms; 16^3 x 32 FP32 343 -> 332 us, with the clover term (8
// x 5) 767 -> 687 us. Four fifths of the rest are the MR steps: 5600 cycles a
// step for the one domain of an SM, 9600 for two.
#include <map>
#include <mutex>

#include "internal.h"
#include "sap_common.cuh"

namespace dwk {

namespace {

template <class C>
struct SapArgs {
    Geom g;
    C diag;
    FieldRef v, x;
    const char* Uimg;             // links of every domain as the shared-memory image of LinkSh
    const unsigned short* faces;  // [ns]: lower-face site | mu << 10 of an inbox slot
    int ns;                       // inbox slots per domain (two per face site and direction)
    char* rho;                    // per rhs: the domains' residuals, site layout of the arithmetic type
    long long rho_rs;
    char* xpart;                  // per rhs: the iterate between cycles, same layout
    long long xpart_rs;
    char* inbox;                  // per rhs: [domain][plane][slot]
    long long inbox_rs;
    const int* jtab;
    int nrhs, nmr;
    int s0, s1, nsweeps;          // sweeps of this launch, sweeps of the application (2 per cycle)
    const char* clov;
    unsigned* bar;                // [2 * DW_MAX_RHS]: barrier and exit counts per rhs (left at zero)
    int* err_host;
};

// a site's spinor in the layout of S32 / S64, read through L2 (other SMs wrote it)
template <class C>
__device__ __forceinline__ void state_load(const char* base, long long V, long long s, cx<C> out[12]) {
    if constexpr (sizeof(C) == 4) {
        const float4* p = reinterpret_cast<const float4*>(base);
#pragma unroll
        for (int q = 0; q < 6; ++q) {
            const float4 v = __ldcg(&p[q * V + s]);
            out[2 * q] = mk<C>(v.x, v.y);
            out[2 * q + 1] = mk<C>(v.z, v.w);
        }
    } else {
        const double2* p = reinterpret_cast<const double2*>(base);
#pragma unroll
        for (int c = 0; c < 12; ++c) {
            const double2 v = __ldcg(&p[c * V + s]);
            out[c] = mk<C>(v.x, v.y);
        }
    }
}

// a half spinor (upper two spin rows) of inbox slot q: 16-byte planes [.][ns]
template <class C>
__device__ __forceinline__ void half_load(const unsigned char* base, int ns, int q, cx<C> h0[3], cx<C> h1[3]) {
    if constexpr (sizeof(C) == 4) {
        const float4* p = reinterpret_cast<const float4*>(base) + q;
        const float4 a = p[0], b = p[ns], c = p[2 * ns];
        h0[0] = mk<C>(a.x, a.y), h0[1] = mk<C>(a.z, a.w), h0[2] = mk<C>(b.x, b.y);
        h1[0] = mk<C>(b.z, b.w), h1[1] = mk<C>(c.x, c.y), h1[2] = mk<C>(c.z, c.w);
    } else {
        const double2* p = reinterpret_cast<const double2*>(base) + q;
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            const double2 a = p[i * ns], b = p[(3 + i) * ns];
            h0[i] = mk<C>(a.x, a.y);
            h1[i] = mk<C>(b.x, b.y);
        }
    }
}
template <class C>
__device__ __forceinline__ void half_store(unsigned char* base, int ns, int q, const cx<C> h0[3], const cx<C> h1[3]) {
    if constexpr (sizeof(C) == 4) {
        float4* p = reinterpret_cast<float4*>(base) + q;
        p[0] = make_float4(h0[0].re, h0[0].im, h0[1].re, h0[1].im);
        p[ns] = make_float4(h0[2].re, h0[2].im, h1[0].re, h1[0].im);
        p[2 * ns] = make_float4(h1[1].re, h1[1].im, h1[2].re, h1[2].im);
    } else {
        double2* p = reinterpret_cast<double2*>(base) + q;
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            p[i * ns] = make_double2(h0[i].re, h0[i].im);
            p[(3 + i) * ns] = make_double2(h1[i].re, h1[i].im);
        }
    }
}

// what a face site sends: SIDE 0, its lower face: (1 + gamma_MU) y; SIDE 1,
// its upper face: U^dagger (1 - gamma_MU) y
template <int MU, class C, class LS>
__device__ __forceinline__ void face_half(int side, const cx<C> y[12], const unsigned char* lsh, int T, int t,
                                          cx<C> k0[3], cx<C> k1[3]) {
    if (side == 0) {
        project<MU, +1, C, true>(y, k0, k1);
    } else {
        cx<C> h0[3], h1[3], u[9];
        project<MU, -1, C, true>(y, h0, h1);
        LS::template load<C>(lsh, T, MU, t, u);
        su3_mul<C, true, true>(u, h0, k0);
        su3_mul<C, true, true>(u, h1, k1);
    }
}

// waits until *cnt reaches target, giving up after about two seconds
__device__ __forceinline__ bool count_wait(const unsigned* cnt, unsigned target) {
    unsigned long long t0 = 0;
    for (unsigned it = 1;; ++it) {
        unsigned v;
        asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(cnt) : "memory");
        if (v >= target) return true;
        if ((it & 255) == 0) {
            const unsigned long long now = global_ns();
            if (t0 == 0)
                t0 = now;
            else if (now - t0 > 2000000000ULL)
                return false;
        }
    }
}

template <int PS, int PL, class C, bool CLOV>
__global__ void __launch_bounds__(256, sizeof(C) == 4 ? 2 : 1) sap_apply_kernel(const __grid_constant__ SapArgs<C> a) {
    constexpr int CP = (sizeof(C) == 4) ? P32 : P64;  // layout of rho and xpart, storage of the clover term
    constexpr int HB = 12 * (int)sizeof(C);           // bytes of a half spinor
    typedef LinkSh<PL> LS;
    extern __shared__ __align__(16) unsigned char smem[];
    const Geom& g = a.g;
    const int T = blockDim.x, ns = a.ns;
    const int rbytes = max((int)sizeof(C) * 24 * T, HB * ns);
    unsigned char* rsh = smem;                                    // inbox, then rho, then y
    unsigned char* lsh = smem + rbytes;                           // links
    C* red = reinterpret_cast<C*>(lsh + (size_t)LS::kBytes * T);  // [32][3]
    unsigned long long* lbar = reinterpret_cast<unsigned long long*>(red + 96);

    const int r = blockIdx.x % a.nrhs;
    const int e = blockIdx.x / a.nrhs;
    if (!rhs_active(a.jtab, r)) return;  // every CTA of this rhs
    const char* vb = field_ptr(a.v, a.jtab, r);
    char* xb = field_ptr(a.x, a.jtab, r);
    char* rho_g = a.rho + (long long)r * a.rho_rs;
    char* xp = (PS == P16 || PS == PB16) ? a.xpart + (long long)r * a.xpart_rs : xb;
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
    const unsigned lbytes = (unsigned)LS::kBytes * (unsigned)T;
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

    bool dead = false;
    for (int sw = a.s0; sw < a.s1; ++sw) {
        const bool first = sw < 2, last = sw >= a.nsweeps - 2;
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
        if (act) {
            if (first)
                load_spinor<PS, C>(vb, g.V, s, rho);
            else
                state_load<C>(rho_g, g.V, s, rho);
        } else {
#pragma unroll
            for (int c = 0; c < 12; ++c) rho[c] = czero<C>();
        }
        // the previous sweep's sends have arrived: fetch the inbox
        bool ok = true;
        if (sw > a.s0) {
            if (tid == 0) ok = count_wait(a.bar + r, ncta * (unsigned)(sw - a.s0));
            __syncthreads();
        }
        if (sw > 0) {
            const unsigned char* src = inb + (long long)dom * HB * ns;
            for (int q = tid; q < HB / 16 * ns; q += T)
                cp_async_word(reinterpret_cast<float4*>(rsh) + q, reinterpret_cast<const float4*>(src) + q);
            cp_async_wait();
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
        // r = rho + 1/2 sum of the hops that enter the domain: first the link
        // products of the forward half spinors, one face site per thread, in place ...
        if (sw > 0) {
            for (int q = tid; q < ns / 2; q += T) {
                const int f = __ldg(a.faces + q), mu = f >> 10;
                const int t = (f & 1023) + (mu == 0 ? g.b[0] - 1 : mu == 1 ? (g.b[1] - 1) * ls1
                                            : mu == 2       ? (g.b[2] - 1) * ls2
                                                            : (g.b[3] - 1) * ls3);
                cx<C> h0[3], h1[3], k0[3], k1[3], u[9];
                half_load<C>(rsh, ns, q, h0, h1);
                LS::template load<C>(lsh, T, mu, t, u);
                su3_mul<C, false, true>(u, h0, k0);
                su3_mul<C, false, true>(u, h1, k1);
                half_store<C>(rsh, ns, q, k0, k1);
            }
            __syncthreads();
            // ... then each site adds what enters through its faces
            if (act) {
                cx<C> acc[12], k0[3], k1[3];
#pragma unroll
                for (int c = 0; c < 12; ++c) acc[c] = czero<C>();
                int off = 0;  // slot of this site's line in direction mu
#define SAP_IN_HOPS(MU, FI)                                     \
    {                                                           \
        const int q = off + (FI);                               \
        if (lx[MU] == g.b[MU] - 1) {                            \
            half_load<C>(rsh, ns, q, k0, k1);                   \
            reconstruct<MU, +1, C, true>(k0, k1, acc);          \
        }                                                       \
        if (lx[MU] == 0) {                                      \
            half_load<C>(rsh, ns, ns / 2 + q, k0, k1);          \
            reconstruct<MU, -1, C, true>(k0, k1, acc);          \
        }                                                       \
        off += g.B / g.b[MU];                                   \
    }
                SAP_IN_HOPS(0, lx[1] + g.b[1] * (lx[2] + g.b[2] * lx[3]))
                SAP_IN_HOPS(1, lx[0] + g.b[0] * (lx[2] + g.b[2] * lx[3]))
                SAP_IN_HOPS(2, lx[0] + g.b[0] * (lx[1] + g.b[1] * lx[3]))
                SAP_IN_HOPS(3, lx[0] + g.b[0] * (lx[1] + g.b[1] * lx[2]))
#undef SAP_IN_HOPS
                const C half = (C)0.5;
#pragma unroll
                for (int c = 0; c < 12; ++c) rho[c] = rho[c] + half * acc[c];
            }
            __syncthreads();  // the inbox makes room for the MR iterate
        }
#pragma unroll
        for (int c = 0; c < 12; ++c) y[c] = czero<C>();

        // MR on D^l y = r^l out of shared memory
        for (int it = 0; it < a.nmr; ++it) {
            rho_store<C>(rsh, T, tid, rho);
            __syncthreads();
            cx<C> p[12];
            C pr_re = 0, pr_im = 0, pp = 0;
            if (act) {
                cx<C> acc[12], psi[12], u[9];
#pragma unroll
                for (int c = 0; c < 12; ++c) acc[c] = czero<C>();
#define SAP_LOC_HOPS(MU, LS_MU)                     \
    {                                               \
        if (lx[MU] + 1 < g.b[MU]) {                 \
            rho_load<C>(rsh, T, tid + LS_MU, psi);  \
            LS::template load<C>(lsh, T, MU, tid, u); \
            hop<MU, +1, C, true>(psi, u, acc);      \
        }                                           \
        if (lx[MU] >= 1) {                          \
            const int tn = tid - LS_MU;             \
            rho_load<C>(rsh, T, tn, psi);           \
            LS::template load<C>(lsh, T, MU, tn, u); \
            hop<MU, -1, C, true>(psi, u, acc);      \
        }                                           \
    }
                SAP_LOC_HOPS(0, 1)
                SAP_LOC_HOPS(1, ls1)
                SAP_LOC_HOPS(2, ls2)
                SAP_LOC_HOPS(3, ls3)
#undef SAP_LOC_HOPS
                // the site's own rho is read back from shared memory (where the
                // neighbours read it) rather than kept in registers over the hops:
                // the 24 registers go to overlapping the hops' loads
                rho_load<C>(rsh, T, tid, rho);
                if constexpr (CLOV) clover_acc<CP, C>(a.clov, g.V, s, rho, acc, (C)-2);  // A rho as -2 A rho in acc
                const C half = (C)0.5;
#pragma unroll
                for (int c = 0; c < 12; ++c) {
                    p[c] = a.diag * rho[c] - half * acc[c];
                    const cx<C> t = cmulc(p[c], rho[c]);
                    pr_re += t.re;
                    pr_im += t.im;
                    pp += p[c].re * p[c].re + p[c].im * p[c].im;
                }
            } else {
#pragma unroll
                for (int c = 0; c < 12; ++c) p[c] = czero<C>();
            }
            block_sum3(pr_re, pr_im, pp, red);
            if (pp > (C)0) {
                const cx<C> alpha = mk<C>(pr_re / pp, pr_im / pp);
#pragma unroll
                for (int c = 0; c < 12; ++c) {
                    y[c] = y[c] + alpha * rho[c];
                    rho[c] = rho[c] - alpha * p[c];
                }
            }
        }

        // the correction's half spinors to the neighbouring domains' inboxes
        if (sw + 1 < a.nsweeps) {
            rho_store<C>(rsh, T, tid, y);
            __syncthreads();
            for (int q = tid; q < ns; q += T) {
                const int side = q >= ns / 2 ? 1 : 0;
                const int f = __ldg(a.faces + q - side * (ns / 2)), mu = f >> 10;
                int t = f & 1023;
                cx<C> yy[12], k0[3], k1[3];
                long long to;
#define SAP_SEND(MU, LS_MU, DST)                                                             \
    {                                                                                        \
        if (side) {                                                                          \
            t += (g.b[MU] - 1) * LS_MU;                                                      \
            to = D[MU] + 1 < g.nb[MU] ? dom + DST : dom - (g.nb[MU] - 1) * DST;              \
        } else {                                                                             \
            to = D[MU] > 0 ? dom - DST : dom + (g.nb[MU] - 1) * DST;                         \
        }                                                                                    \
        rho_load<C>(rsh, T, t, yy);                                                          \
        face_half<MU, C, LS>(side, yy, lsh, T, t, k0, k1);                                   \
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
                half_store<C>(inb + to * HB * ns, ns, q, k0, k1);
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
        // x^l <- x^l + y^l; rho^l is kept for the next visit
        if (act) {
            if (!first) {
                cx<C> xo[12];
                state_load<C>(xp, g.V, sc, xo);
#pragma unroll
                for (int c = 0; c < 12; ++c) y[c] = y[c] + xo[c];
            }
            if (last) {
                store_spinor<PS, C>(xb, g.V, sc, y);
            } else {
                store_spinor<CP, C>(xp, g.V, sc, y);
                store_spinor<CP, C>(rho_g, g.V, sc, rho);
            }
        }
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

template <int PS, int PL, class C>
int sap_apply_t(const Geom& g, double m0, FieldRef v, FieldRef x, const SapWork& w, const int* jtab, int nrhs,
                int ncycles, int nmr, cudaStream_t st, const ClovRef* cl, Profiler* prof, double bytes_first,
                double bytes_next) {
    const int threads = sap_threads(g, 0);
    const size_t smem = (size_t)sap_apply_smem(PS, PL, g);
    const void* fn = cl ? (const void*)sap_apply_kernel<PS, PL, C, true> : (const void*)sap_apply_kernel<PS, PL, C, false>;
    // per device and CTA shape: the shared-memory limit is raised once, and the
    // CTAs that the device holds at a time are asked for once
    static std::mutex mu;
    static std::map<std::pair<int, std::pair<const void*, std::pair<int, size_t>>>, int> resident;
    int dev = 0, fit = 0;
    DW_CUDA_TRY(cudaGetDevice(&dev));
    {
        std::lock_guard<std::mutex> lock(mu);
        const auto key = std::make_pair(dev, std::make_pair(fn, std::make_pair(threads, smem)));
        auto it = resident.find(key);
        if (it == resident.end()) {
            int sms = 0, per = 0;
            DW_CUDA_TRY(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024));
            DW_CUDA_TRY(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
            DW_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, fn, threads, smem));
            it = resident.emplace(key, sms * per).first;
        }
        fit = it->second;
    }
    SapArgs<C> a;
    a.g = g;
    a.diag = (C)(4.0 + m0);
    a.v = v;
    a.x = x;
    a.Uimg = w.Uimg;
    a.faces = w.faces;
    a.ns = sap_inbox_slots(g);
    a.rho = w.rho;
    a.rho_rs = w.rho_rs;
    a.xpart = w.xpart;
    a.xpart_rs = w.xpart_rs;
    a.inbox = w.inbox;
    a.inbox_rs = w.inbox_rs;
    a.jtab = jtab;
    a.nrhs = nrhs;
    a.nmr = nmr;
    a.nsweeps = 2 * ncycles;
    a.clov = cl ? ((sizeof(C) == 4) ? cl->a32 : cl->a64) : nullptr;
    a.bar = w.bar;
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
    if ((long long)cfg.gridDim.x <= fit) {
        attr[0].id = cudaLaunchAttributeCooperative;
        attr[0].val.cooperative = 1;
        a.s0 = 0;
        a.s1 = a.nsweeps;
        ProfScope ps(prof, "sap_sweep", 2.0 * bytes_first + (a.nsweeps - 2) * bytes_next, a.nsweeps);
        DW_CUDA_TRY(cudaLaunchKernelExC(&cfg, fn, args));
        DW_LAUNCH_CHECK();
        return DW_OK;
    }
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    for (int sw = 0; sw < a.nsweeps; ++sw) {
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
    const int c = (pspin == P64) ? 8 : 4, T = sap_threads(g, 0);
    const int body = std::max(c * 24 * T, c * 12 * sap_inbox_slots(g));
    return body + (int)(sap_link_image_bytes(plink, g, T) / g.ndom) + c * 96 + 16;
}

// Domains of at most 256 sites whose inbox is no larger than a double-precision
// field (the scratch that a solve has at hand) and fits in shared memory.
bool sap_apply_fits(int prec, const Geom& g) {
    const long long c = (prec == P64) ? 8 : 4;
    return g.B <= 256 && 12 * c * sap_inbox_slots(g) <= 192LL * g.B && sap_apply_smem(prec, prec, g) <= 227 * 1024;
}

void sap_faces(const Geom& g, std::vector<unsigned short>* out) {
    out->clear();
    int ls = 1;
    for (int mu = 0; mu < 4; ++mu) {
        for (int t = 0; t < g.B; ++t)
            if ((t / ls) % g.b[mu] == 0) out->push_back((unsigned short)(t | (mu << 10)));
        ls *= g.b[mu];
    }
}

int launch_sap_apply(int prec, const Geom& g, double m0, FieldRef v, FieldRef x, const SapWork& w, const int* jtab,
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
