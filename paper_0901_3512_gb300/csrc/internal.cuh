// Internal declarations shared by the library's translation units.
//
// Device data layout (GB300: 32-wide warps, 128-byte lines; every kernel
// below maps one thread to one lattice site so that neighbouring threads
// touch neighbouring addresses):
//   spinor       element k = 3*spin + colour (0..11) of site s at flat complex index
//                ((k/2)*V + s)*2 + k%2: six "pair" planes, each site's two complex
//                entries of a plane adjacent (one 16-byte load in FP32, 32 bytes in FP64);
//                the same flat order in FP64 (double2) and FP32 (float2)
//   links        T2      [4][9][V]    U_mu(x)[a][b] at [(mu*9 + 3a + b)*V + s]
// A basis vector of V is one spinor in the same flat order, in the storage
// type of the precision mode (double2, float2 or bf16x2 per complex entry).
#pragma once

#include <atomic>

#include <cuda_runtime.h>
#include <cuda_bf16.h>
#include <stdint.h>
#include <stdio.h>
#include <string>

#include "../../include/seedcg.h"
#include "device_once.h"

namespace seedcg {

// ----------------------------------------------------------------------------
// errors
// ----------------------------------------------------------------------------
struct Error {
    seedcg_status code;
    std::string msg;
};

#define SEEDCG_CUDA_TRY(expr)                                                              \
    do {                                                                                   \
        cudaError_t e_ = (expr);                                                           \
        if (e_ != cudaSuccess) {                                                           \
            throw ::seedcg::Error{e_ == cudaErrorMemoryAllocation ? SEEDCG_ERR_OOM         \
                                                                  : SEEDCG_ERR_CUDA,       \
                                  std::string(#expr) + ": " + cudaGetErrorString(e_)};     \
        }                                                                                  \
    } while (0)

constexpr int kMaxGridY = 65535;   // the most blocks of a grid in y: fields side by side beyond it take another launch

// every kernel launch site ends with this: it checks the launch and counts it
extern std::atomic<unsigned long long> g_kernel_launches;
#define SEEDCG_CHECK_LAUNCH()                                                              \
    do {                                                                                   \
        ::seedcg::g_kernel_launches.fetch_add(1, std::memory_order_relaxed);               \
        SEEDCG_CUDA_TRY(cudaGetLastError());                                               \
    } while (0)

// Dynamic shared memory above 48 KB for a kernel, on the device that is current (the attribute belongs to a device)
template <auto Kernel>
inline void allow_smem(size_t bytes) {
    static DeviceOnce once;
    int dev = 0;
    SEEDCG_CUDA_TRY(cudaGetDevice(&dev));
    once.run(dev, [&]() {
        SEEDCG_CUDA_TRY(cudaFuncSetAttribute(Kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes));
    });
}

// Programmatic dependent launch for the kernels of the iteration loops, which are a few
// microseconds each: launch_pdl lets the next kernel of the stream be placed on the SMs while the previous
// one still runs, and pdl_enter, the first statement of every such kernel, waits until that one is complete
// and visible, then lets the kernel after it come up.  Every kernel launched this way has to call it on every
// path: one that returned without waiting would let its successor overtake its predecessor.
// Such a kernel is resident while its predecessor writes, so what it reads is not constant during its life: only links
// and tables written long before come through __ldg or a __restrict__ pointer (which let the compiler take the
// read-only path, or move a load above the wait); fields, partials and coefficients are loaded plainly, and
// __restrict__ stays on outputs that the kernel never reads.
#ifdef __CUDACC__
__device__ __forceinline__ void pdl_enter() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
// Only where the kernels are short, `entries` complex entries per launch: on 10x6x14x12 with 5 systems a solve
// takes 37.0 ms without it and 33.4 ms with it, but at 16^3 x 32 the early blocks take slots that the running
// kernel's own blocks would have used (250.6 against 254.1 ms; even-odd 113.1 against 115.5 ms).
inline bool pdl_for(long entries) { return entries <= 12L * 49152; }
// The launches of one FP32 application, `entries` over all of the fields of a launch: two to four kernels in a row, where
// the early launch hides the next one's start. us without -> with it, M / M by single-field kernels / A^dag A:
//   8^3 x 16:  12 fields 48.4 -> 43.8 / 45.1 -> 42.6 / 69.4 -> 70.3; 48 fields 120.3 -> 115.2 / 113.2 -> 106.8 / 116.6 -> 107.3
//   12^3 x 24:  6 fields 96.9 -> 94.1 / 89.3 -> 83.8 / 112.2 -> 105.1; 18 fields 210.2 -> 206.6 / 193.4 -> 187.3 / 247.2 -> 238.4
//   16^3 x 32:  2 fields 93.5 -> 89.0 / 92.7 -> 88.2 / 172.5 -> 167.1; 12 fields 392.6 -> 390.2 / 377.3 -> 367.7 / 395.1 -> 385.2
// The gain ends at the last (19 M entries): the line.
inline bool pdl_for_apply(long entries) { return entries <= 12L * 1572864; }
template <typename... P, typename... A>
void launch_pdl(bool early, void (*kernel)(P...), dim3 grid, int block, size_t smem, cudaStream_t st, A... args) {
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(block);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cfg.attrs = at;
    cfg.numAttrs = early ? 1 : 0;
    SEEDCG_CUDA_TRY(cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...));
    g_kernel_launches.fetch_add(1, std::memory_order_relaxed);
}
#endif

// ----------------------------------------------------------------------------
// complex helpers on CUDA vector types
// ----------------------------------------------------------------------------
template <typename R> struct Cx;
template <> struct Cx<double> { using T = double2; };
template <> struct Cx<float> { using T = float2; };
template <typename R> using cx_t = typename Cx<R>::T;

template <typename R> __host__ __device__ __forceinline__ cx_t<R> mk(R re, R im) {
    cx_t<R> z; z.x = re; z.y = im; return z;
}
template <typename C> __host__ __device__ __forceinline__ C cadd(C a, C b) { a.x += b.x; a.y += b.y; return a; }
template <typename C> __host__ __device__ __forceinline__ C csub(C a, C b) { a.x -= b.x; a.y -= b.y; return a; }
// a * b
template <typename C> __host__ __device__ __forceinline__ C cmul(C a, C b) {
    C z; z.x = a.x * b.x - a.y * b.y; z.y = a.x * b.y + a.y * b.x; return z;
}
// acc + a * b
template <typename C> __host__ __device__ __forceinline__ C cfma(C a, C b, C acc) {
    acc.x = fma(a.x, b.x, fma(-a.y, b.y, acc.x));
    acc.y = fma(a.x, b.y, fma(a.y, b.x, acc.y));
    return acc;
}
// acc + conj(a) * b
template <typename C> __host__ __device__ __forceinline__ C cfma_conj(C a, C b, C acc) {
    acc.x = fma(a.x, b.x, fma(a.y, b.y, acc.x));
    acc.y = fma(a.x, b.y, fma(-a.y, b.x, acc.y));
    return acc;
}
// i * a
template <typename C> __host__ __device__ __forceinline__ C ci(C a) { C z; z.x = -a.y; z.y = a.x; return z; }
template <typename C, typename R> __host__ __device__ __forceinline__ C cscale(C a, R s) { a.x *= s; a.y *= s; return a; }

// ----------------------------------------------------------------------------
// lattice geometry
// ----------------------------------------------------------------------------
struct Geom {
    int L[4];        // Lx, Ly, Lz, Lt
    int vol;         // sites
    int stride[4];   // 1, Lx, Lx*Ly, Lx*Ly*Lz
};

inline Geom make_geom(const int dims[4]) {
    Geom g;
    for (int i = 0; i < 4; i++) g.L[i] = dims[i];
    g.stride[0] = 1;
    g.stride[1] = dims[0];
    g.stride[2] = dims[0] * dims[1];
    g.stride[3] = dims[0] * dims[1] * dims[2];
    g.vol = g.stride[3] * dims[3];
    return g;
}

// One gauge field for the FP64 operator (fixhop.cuh): the links in fixed point,
// L = -kappa U 2^k with the antiperiodic sign, [4][9][V] (re hi, re lo, im hi, im lo),
// and the FP64 links for what the fixed point cannot take (ok = 0: for every site; there is no L then).
struct FixDev {
    Geom g;
    const int4* L;
    const double2* u;
    double kappa;
    int k;
    int ok;
};

// ----------------------------------------------------------------------------
// device buffers
// ----------------------------------------------------------------------------
// Frees the scratch that handles keep between calls (KeptScratch) and do not use now; true if there was any.
bool give_back_scratch();

// Owning device allocation: freed by the destructor (or release()); move-only.
struct DevBuf {
    void* p = nullptr;
    size_t bytes = 0;
    DevBuf() = default;
    DevBuf(const DevBuf&) = delete;
    DevBuf& operator=(const DevBuf&) = delete;
    DevBuf(DevBuf&& o) noexcept : p(o.p), bytes(o.bytes) {
        o.p = nullptr;
        o.bytes = 0;
    }
    DevBuf& operator=(DevBuf&& o) noexcept {
        if (this != &o) {
            release();
            p = o.p;
            bytes = o.bytes;
            o.p = nullptr;
            o.bytes = 0;
        }
        return *this;
    }
    ~DevBuf() { release(); }
    void ensure(size_t n) {
        if (n <= bytes) return;
        release();
        cudaError_t e = cudaMalloc(&p, n);
        if (e == cudaErrorMemoryAllocation) {
            cudaGetLastError();   // not an error of the next launch
            if (give_back_scratch()) e = cudaMalloc(&p, n);
        }
        if (e != cudaSuccess) {
            cudaGetLastError();
            p = nullptr;
            throw Error{e == cudaErrorMemoryAllocation ? SEEDCG_ERR_OOM : SEEDCG_ERR_CUDA,
                        "cudaMalloc of " + std::to_string(n) + " bytes: " + cudaGetErrorString(e)};
        }
        bytes = n;
    }
    void release() {
        if (p) cudaFree(p);
        p = nullptr;
        bytes = 0;
    }
    template <typename T> T* as() const { return reinterpret_cast<T*>(p); }
};

// Scratch that a handle keeps between calls, so that a repeated call does not pay for cudaMalloc and cudaFree (at 36 MB
// they took 175 us of a 390 us call).  All handles of the process together keep at most kKeptBytes (what M takes on twelve FP64 fields
// of 16^3 x 32 is 302 MB; a call that needs more frees its scratch when it returns, as every call did when nothing was
// kept), and what is kept never stands in the way of an allocation of this library: DevBuf::ensure gives it back first.
// Safe between threads that use different handles.
class KeptScratch {
    DevBuf buf_;
    bool busy_ = false;
    friend bool give_back_scratch();

public:
    static constexpr size_t kKeptBytes = (size_t)512 << 20;
    KeptScratch();
    ~KeptScratch();
    KeptScratch(const KeptScratch&) = delete;
    KeptScratch& operator=(const KeptScratch&) = delete;
    class Use {   // the scratch for one call, which ends with its device work
        KeptScratch& s_;
        int exceptions_;   // in flight when the call began

    public:
        Use(KeptScratch& s, size_t bytes);
        ~Use();
        Use(const Use&) = delete;
        Use& operator=(const Use&) = delete;
        template <typename T> T* as() const { return s_.buf_.as<T>(); }
    };
};

// ----------------------------------------------------------------------------
// launchers implemented in dslash.cu
// ----------------------------------------------------------------------------
// canonical complex128 AoS [n][V][12] <-> internal
void to_internal_f64(const double* in, double2* out, int vol, int n, cudaStream_t s);
void from_internal_f64(const double2* in, double* out, int vol, int n, cudaStream_t s);
void to_internal_f32(const double* in, float2* out, int vol, int n, cudaStream_t s);
void gauge_to_internal(const double* in, double2* u64, float2* u32, int vol, cudaStream_t s);

// FP32: out = D in (dag = 0) or D^dag in (dag = 1) for n fields at in + r*12*V; out: internal
// (OutF32) or the boundary's complex128 [n][V][4][3] (OutF64, widened at the store)
struct OutF32 { float2* p; };
struct OutF64 { double* p; int wide; };   // wide: p is 32-byte aligned (make_out_f64)
inline OutF64 make_out_f64(double* p) { return OutF64{p, (reinterpret_cast<uintptr_t>(p) & 31) == 0}; }
// links staged once per tile of sites; fixed: the default tile shape, never timing alternatives
template <typename Out>
void dslash_mrhs_f32(const Geom& g, const float2* u, float kappa, int dag, int n, const float2* in, Out out,
                     bool fixed, cudaStream_t s);

// op 0 = D, 1 = D^dag, 2 = M on the boundary's fields in FP32 arithmetic: in is rounded into `work` (n internal
// fields; 2 n for op 2), the last operator writes out.  multi = 0: links from global memory.
void apply_spinors_f32(const Geom& g, const float2* u, float kappa, int op, int multi, bool fixed, int n,
                       const double* in, double* out, float2* work, cudaStream_t s);

// FP64 operator in fixed point (fixed.cu): out = D in or D^dag in for n fields
void dslash_f64(const FixDev& F, int dag, int n, const double2* in, double2* out, cudaStream_t s);
// the same on the boundary's complex128 fields [n][V][4][3], without a layout pass: op 0 = D, 1 = D^dag,
// 2 = M (tmp: n internal fields of scratch, op 2 only)
void apply_spinors_f64(const FixDev& F, int op, int n, const double* in, double* out, double2* tmp, cudaStream_t s);
// A, A^dag or A^dag A on complex128 half fields (te: n half vectors of scratch; tmp: n more, op 2 only)
void apply_eo_spinors_f64(const FixDev& F, int op, int n, const double* in, double* out, double2* te, double2* tmp,
                          cudaStream_t s);
// the scale k of a handle's links in fixed point, and whether they fit it (synchronises); the links themselves
void fix_scale(const Geom& g, const double2* u, double kappa, int* k, int* ok, cudaStream_t s);
void fix_links(const Geom& g, const double2* u, double kappa, int k, int4* L, cudaStream_t s);

// even-odd preconditioned system (fixed.cu), FP64 half vectors in the internal layout:
// out_r = A x_r (dag = 0) or A^dag x_r, A = 1 - kappa^2 H_oe H_eo, n fields (te: n even half
// vectors of scratch; out may be x)
void eo_apply_a_f64(const FixDev& F, int dag, int n, const double2* x, double2* te, double2* out, cudaStream_t st);
// out_r = A^dag A x_r (te: n even half vectors of scratch)
void eo_apply_mdag_m_f64(const FixDev& F, int n, const double2* x, double2* te, double2* out, cudaStream_t st);
// phi = eta_o + kappa H_oe eta_e for n full fields eta
void eo_source_f64(const FixDev& F, int n, const double2* eta, double2* phi, cudaStream_t st);
// half[r] = the parity-p sites of full[r] for n fields
void eo_gather_f64(const Geom& g, int p, int n, const double2* full, double2* half, cudaStream_t st);
// full x from x_o: x_e = eta_e + kappa H_eo x_o, for n fields
void eo_reconstruct_f64(const FixDev& F, int n, const double2* x_odd, const double2* eta, double2* x,
                        cudaStream_t st);

}  // namespace seedcg
