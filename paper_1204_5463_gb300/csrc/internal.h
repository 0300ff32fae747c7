// Host-side internals of the library: the context object and the launchers
// of the CUDA kernels (declared here, defined in the .cu files).
#pragma once

#include <cuda_runtime.h>

#include <atomic>

#include <complex>
#include <string>
#include <vector>

#include "../../include/dwsolve.h"
#include "common.cuh"

namespace dwk {

typedef std::complex<double> zd;

// thread-local error message behind dw_last_error()
void set_error(const std::string& msg);
int fail(int code, const std::string& msg);

#define DW_CUDA_TRY(expr)                                                                       \
    do {                                                                                        \
        cudaError_t _e = (expr);                                                                \
        if (_e != cudaSuccess)                                                                  \
            return ::dwk::fail(DW_ECUDA, std::string(#expr) + ": " + cudaGetErrorString(_e));   \
    } while (0)

// Largest lattice a context accepts: spinor element indices (24 reals per
// site) stay below 2^31, so device code may use 32-bit site arithmetic.
constexpr long long kMaxSites = (1LL << 31) / 24;

// V = d1 d2 d3 d4 for caller-supplied extents, checked as it is formed: every
// extent >= 2 and the running product <= max_sites (so the product can neither
// overflow nor wrap to a small value). Returns false with *V untouched otherwise.
inline bool lattice_volume(const int* dims, long long max_sites, long long* V) {
    long long v = 1;
    for (int j = 0; j < 4; ++j) {
        if (dims[j] < 2 || dims[j] > max_sites) return false;
        v *= dims[j];
        if (v > max_sites) return false;
    }
    *V = v;
    return true;
}

// Every kernel launch of the library is followed by DW_LAUNCH_CHECK(): it
// counts the launch (dw_kernel_launches()) and turns a launch error into DW_ECUDA.
void count_launch();
#define DW_LAUNCH_CHECK()          \
    do {                           \
        ::dwk::count_launch();     \
        DW_CUDA_TRY(cudaGetLastError()); \
    } while (0)

// A device allocation owned by the library (grown on demand, freed with the owner).
struct DevBuf {
    void* p = nullptr;
    size_t bytes = 0;
    cudaStream_t st = nullptr;  // allocations are stream-ordered on the owner's stream
    int ensure(size_t n);
    void release();
    template <class T>
    T* as() const { return reinterpret_cast<T*>(p); }
    ~DevBuf() { release(); }
};

// Per-kernel-class timing, collected with CUDA events on the library stream
// while profiling is switched on.
struct KernelProfile {
    std::string name;
    long long launches = 0;  // units of work: launches, or the SAP sweeps that one launch runs
    double total_ms = 0.0;
    double bytes = 0.0;  // algorithmic bytes summed over launches
    std::vector<std::pair<cudaEvent_t, cudaEvent_t>> pending;
    std::vector<double> pending_bytes;
    std::vector<int> pending_count;
};

struct Profiler {
    bool on = false;
    std::vector<KernelProfile> k;
    std::vector<cudaEvent_t> pool;  // recycled events (creation is not free)
    cudaStream_t stream = nullptr;
    cudaEvent_t take();
    int begin(const char* name, double bytes, cudaEvent_t* start_out, int* idx, int count = 1);
    void end(int idx, cudaEvent_t start);
    void drain();  // turn pending event pairs into totals (synchronises)
    void reset();
    ~Profiler();
};

// RAII helper: times the launches issued in its scope as one entry.
struct ProfScope {
    Profiler* p;
    int idx = -1;
    cudaEvent_t start = nullptr;
    ProfScope(Profiler* prof, const char* name, double bytes, int count = 1) : p(prof) {
        if (p && p->on) p->begin(name, bytes, &start, &idx, count);
    }
    ~ProfScope() {
        if (p && p->on && idx >= 0) p->end(idx, start);
    }
};

struct Workspace;                    // Krylov workspace of the solver (solver.cpp)
void release_workspace(Workspace* w);

}  // namespace dwk

namespace dwk {
// The clover term of a context: FP64 storage (double [72][V]) for double and
// double-float arithmetic, FP32 storage (float4 [18][V]) for float arithmetic.
struct ClovRef {
    const char* a64;
    const char* a32;
};

// An int in host-mapped pinned memory that kernels set to report a bounded
// wait that gave up; the host reads it after synchronising the stream.
struct HostFlag {
    int* h = nullptr;  // host address
    int* d = nullptr;  // device address
    int ensure();
    ~HostFlag();
};
}  // namespace dwk

struct dw_ctx {
    dwk::Geom g;
    double m0 = 0.0;
    cudaStream_t stream = nullptr;
    int device = 0;
    bool have_gauge = false;
    dwk::DevBuf U[5];           // gauge field per storage precision (P64, P32, P16, PB16, PDF)
    bool U_ready[5] = {false, false, false, false, false};
    dwk::DevBuf work_in, work_out, work_aux;  // conversions in dw_apply / sap_precondition
    dwk::Profiler prof;
    dwk::Workspace* ws = nullptr;  // solver workspace, kept between solves
    double csw = 0.0;               // clover coefficient (0: plain Wilson operator)
    dwk::DevBuf clov64, clov32;     // clover term, FP64 [72][V] and FP32 float4 [18][V]
    dwk::ClovRef clov{nullptr, nullptr};
    dwk::DevBuf Uimg[4];            // SAP links per domain as shared-memory images (per storage precision)
    bool Uimg_ready[4] = {false, false, false, false};
    dwk::HostFlag sap_err;          // set by a SAP kernel whose bounded wait gave up
    unsigned long long sap_wait_ns = 2000000000ULL;  // SapWork::kWait, unless dw_debug_sap_wait changed it
    std::atomic<int> cancel{0};     // set by dw_cancel; the running solve stops before its next step
    const dwk::ClovRef* clover() const { return csw != 0.0 ? &clov : nullptr; }
};

namespace dwk {

// gauge field in the requested storage precision (converted from FP64 on first use)
int gauge_for(dw_ctx* ctx, int prec, const char** out);

// ----- dw.cu ---------------------------------------------------------------
// canonical FP64 <-> internal layout of nrhs fields; scale (device, one double
// per rhs, may be null) multiplies every value on the way
int launch_to_internal(int prec, const double* canon, char* out, long long V, int nrhs, cudaStream_t st,
                       const double* scale = nullptr);
int launch_from_internal(int prec, const char* in, double* canon, long long V, int nrhs, cudaStream_t st,
                         const double* scale = nullptr);
int launch_gauge_convert(int prec, const double* Ucanon, char* out, long long V, cudaStream_t st);
int launch_link_convert(int prec, const char* U64, char* out, long long V, cudaStream_t st);

// out = D in  (sub == nullptr)   or   out = sub - D in  (sub: FP64 field, PO must be P64);
// with cl, D includes the clover term
int launch_dw(int pin, int pout, int plink, const Geom& g, double m0, FieldRef in, FieldRef out, const char* U,
              RhsCols jtab, int nrhs, const FieldRef* sub, cudaStream_t st, const ClovRef* cl = nullptr);
// out (caller's FP64 layout, nrhs fields) = D in, all in storage precision prec (P64, P32, P16, PB16)
int launch_dw_out(int prec, const Geom& g, double m0, const char* in, double* out, const char* U, int nrhs,
                  cudaStream_t st, const ClovRef* cl = nullptr);
// ----- clover.cu -----------------------------------------------------------
int launch_clover_compute(const Geom& g, const char* U64, double csw, double* A64, float4* A32, cudaStream_t st);

// ----- sap.cu --------------------------------------------------------------
// One colour half-sweep of SAP (Algorithm 2) on every domain of `colour`:
// r = v - D x (full operator), nmr MR steps on D^l y = r, x += y.
// mode 0: x == 0 everywhere (r = v, x = y); 1: x == 0 on this colour; 2: general.
// Uimg: the links of every domain packed by launch_sap_link_image (the sweep reads
// its links only there); err_host: HostFlag::d, set if a link copy did not complete.
int launch_sap_sweep(int pspin, int plink, const Geom& g, double m0, FieldRef v, FieldRef x, const char* Uimg,
                     RhsCols jtab, int nrhs, int colour, int nmr, int mode, cudaStream_t st,
                     const ClovRef* cl, int* err_host);
int sap_smem_bytes(int pspin, int plink, const Geom& g);
// CTA size of the SAP kernels: the domain volume rounded up to a warp multiple
int sap_threads(const Geom& g);
size_t sap_link_image_bytes(int plink, const Geom& g);
int launch_sap_link_image(int plink, const Geom& g, const char* U, char* img, cudaStream_t st);
// links of precision prec in both layouts (the image is packed on first use, after
// dw_set_gauge and after a wait that gave up), and the error flag
int sap_links_for(dw_ctx* ctx, int prec, const char** U, char** img);
// ----- sap_apply.cu --------------------------------------------------------
// z = M v with the domains' halos exchanged as half spinors (sap_apply.cu), for
// domains that sap_apply_fits accepts. inbox: scratch per right-hand side.
struct SapWork {
    char* Uimg;  // of launch_sap_apply_image, with the face table and the counters behind the links
    char* inbox;
    long long inbox_rs;
    int* err;
    unsigned long long wait_ns;  // limit of a wait for the previous sweep
    static constexpr unsigned long long kWait = 2000000000ULL;
};
bool sap_apply_fits(int prec, const Geom& g);
int sap_apply_smem(int pspin, int plink, const Geom& g);
int sap_inbox_slots(const Geom& g);
// the packed links, the table of inbox slots and the barrier counters, at zero (they
// are left at zero by an application, except by one whose wait gave up)
size_t sap_apply_image_bytes(int prec, const Geom& g);
unsigned short* sap_apply_faces(int prec, const Geom& g, char* img);
unsigned* sap_apply_counters(int prec, const Geom& g, char* img);
int launch_sap_apply_image(int prec, const Geom& g, const char* U, char* img, cudaStream_t st);
int launch_sap_apply(int prec, const Geom& g, double m0, FieldRef v, FieldRef x, const SapWork& w, RhsCols jtab,
                     int nrhs, int ncycles, int nmr, cudaStream_t st, const ClovRef* cl, Profiler* prof,
                     double bytes_first, double bytes_next);
// Scratch of one application and right-hand side: at most a double-precision
// field (192 bytes per site).
size_t sap_inbox_bytes(int prec, const Geom& g);
// the whole application, nact of the nrhs right-hand sides active: by
// launch_sap_apply where the domain fits, else sweep by sweep (the scratch is
// then unused); inbox: scratch of the stride given. Uimg: the image
// of sap_links_for, packed (if it had to be) before at least one ordinary launch
// or copy of the stream: the first sweep is launched programmatically and reads the
// image before it waits for the kernel in front of it, so that kernel must not
// be the one that writes the image.
int sap_run(dw_ctx* ctx, int prec, char* Uimg, FieldRef v, FieldRef x, char* inbox,
            long long inbox_rs, RhsCols jtab, int nrhs, int nact, int ncycles, int nmr);
// after the stream was synchronised: DW_ETIMEOUT if a SAP kernel's bounded wait gave up
int sap_check(dw_ctx* ctx);

// ----- blas.cu -------------------------------------------------------------
// Outer vectors: flat arrays of 16-byte complex elements, format vp = P64
// (double2) or PDF (double-float float4). Column addressing as for FieldRef,
// in elements.
struct VecRef {
    double2* base;
    long long rhs_stride;  // in elements
    long long col_stride;  // in elements
    int col_off;
};
// out[r][i] = <V_i, w>  (i < nv[r]),  out[r][nvmax] = ||w||^2 ; nv = jtab[r] + nv_off (or nv_off)
// nv_active: the largest number of basis vectors any rhs has in this launch
// (sizes the grid); nvmax: the row length of partial/out minus one
// cnt: zeroed counters (left zeroed), kDotCounters per rhs: the last CTA of each
// group of vectors sums the group's partial rows itself. cols (device, one int per rhs, may be null) receives the
// column table for the multi-axpy after it: reading the table from memory, that
// kernel's loop is 643 us where every form with the table in its parameters is
// 664 to 863 us (12 rhs, 16 vectors on average, 16^3 x 32)
constexpr int kDotCounters = 8;
int launch_multidot(int vp, VecRef Vb, VecRef w, long long n, RhsCols jtab, int nv_off, int nvmax, int nv_active,
                    int nrhs, double2* partial, int nblk, double2* out, cudaStream_t st, unsigned* cnt, int* cols = nullptr);
// w -= sum_i coef[r][i] V_i (i < nv[r]);  out_norm2[r] = ||w||^2 after the update;
// cnt: one zeroed counter per rhs (left zeroed); nullptr: a separate reduction launch; jtab: the device table of the multi-dot
int launch_multiaxpy(int vp, VecRef Vb, VecRef w, long long n, const int* jtab, int nv_off, int nrhs,
                     const double2* coef, int coef_ld, double2* partial, int nblk, double* out_norm2,
                     cudaStream_t st, unsigned* cnt = nullptr);
// dst = w / sqrt(norm2[r]) per site; if plow >= 0 also written to `low` in spinor storage plow
int launch_normalize(int vp, VecRef w, VecRef dst, long long V, RhsCols jtab, int nrhs, const double* norm2,
                     int plow, FieldRef low, cudaStream_t st);
// in place, per element: X_c = sum_i X_i Q[r][i][c]  (c < kout, i < nin), X in precision prec
// (scaled FP16/BF16 storage goes through `scratch`, nrhs * kout columns, and is copied back)
int launch_rotate(int prec, char* X, long long rhs_stride, long long col_stride, long long V, int nrhs,
                  const int* active, int nin, int kout, const double2* Q, int qld, char* scratch,
                  cudaStream_t st);
// x[r] += sum_i Z_i eta[r][i]  (i < nz[r]), Z in precision prec, x outer format vx;
// z_rs, z_cs, x_rs in bytes
int launch_xupdate(int prec, int vx, const char* Z, long long z_rs, long long z_cs, double2* x, long long x_rs,
                   long long V, int nrhs, const int* nz, const double2* eta, int eta_ld, cudaStream_t st);
// out[r] = ||a[r]||^2
int launch_norm2(int vp, const double2* a, long long rs, long long n, int nrhs, double2* partial, int nblk,
                 double* out, cudaStream_t st);
// convert a spinor field between storage precisions for a set of rhs
int launch_convert(int pin, int pout, FieldRef in, FieldRef out, long long V, RhsCols jtab, int nrhs,
                   cudaStream_t st);
// dst = a[r] * src  (outer vectors)
int launch_scale(int vp, const double2* src, double2* dst, long long rs, long long n, int nrhs, const double* a,
                 cudaStream_t st);
int launch_zero(void* p, size_t bytes, cudaStream_t st);

int blas_nblk(long long n);

// ----- solver.cpp ----------------------------------------------------------
// validated solve; it stops with DW_ECANCELLED before an Arnoldi step once
// *cancel is non-zero (cancel may be null)
int solve_checked(dw_ctx* ctx, const double* b, double* x, const dw_solver_params* P, dw_stats* S,
                  const std::atomic<int>* cancel);
int solve(dw_ctx* ctx, const double* b, double* x, const dw_solver_params* P, dw_stats* S,
          const std::atomic<int>* cancel);
// the per-cycle residual history of the last solve on ctx (see dw_residual_history)
int residual_history(dw_ctx* ctx, int rhs, double* out, int max, int* n);
// the basis of the last cycle of the last solve on ctx (see dw_debug_basis)
int debug_basis(dw_ctx* ctx, int rhs, double* V_out, double* Z_out, double* H_out, int max_cols, int* ncols);

}  // namespace dwk
