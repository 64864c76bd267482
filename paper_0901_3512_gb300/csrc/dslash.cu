// FP32 Wilson dslash kernels (single- and multi-right-hand-side; FP64: fixed.cu)
// and the layout transforms between the boundary's complex128 AoS and the
// internal site-fastest layouts.
#include <algorithm>
#include <cstdio>
#include <cstdlib>
#include <map>
#include <mutex>
#include <string>
#include <type_traits>

#include "internal.cuh"
#include "wilson.cuh"
#include "reduce.cuh"

namespace seedcg {

namespace {

constexpr int kThreads = 128;

inline int blocks_for(long n, int threads) { return (int)((n + threads - 1) / threads); }

// ---------------------------------------------------------------------------
// layout transforms
// ---------------------------------------------------------------------------
__global__ void k_to_internal_f64(const double2* __restrict__ in, double2* __restrict__ out,
                                  int vol, int n) {
    long t = blockIdx.x * (long)blockDim.x + threadIdx.x;
    if (t >= (long)vol * n) return;
    int r = (int)(t / vol), s = (int)(t % vol);
    const double2* src = in + ((size_t)r * vol + s) * 12;
    double2* dst = out + (size_t)r * 12 * vol;
#pragma unroll
    for (int k = 0; k < 12; k++) dst[sidx(k, s, vol)] = src[k];
}

// (with 16-byte stores every 32-byte sector is written twice: 12 fields of 16^3 x 32 take 196 us, in whole
// sectors 88; `wide`: out is 32-byte aligned, and so is every spinor)
__global__ void k_from_internal_f64(const double2* __restrict__ in, double2* __restrict__ out,
                                    int vol, int n, int wide) {
    long t = blockIdx.x * (long)blockDim.x + threadIdx.x;
    if (t >= (long)vol * n) return;
    int r = (int)(t / vol), s = (int)(t % vol);
    const double2* src = in + (size_t)r * 12 * vol;
    double2* dst = out + ((size_t)r * vol + s) * 12;
    double2 z[12];
#pragma unroll
    for (int k = 0; k < 12; k++) z[k] = src[sidx(k, s, vol)];
#pragma unroll
    for (int k = 0; k < 12; k += 2) {
        if (wide) {
            asm volatile("st.global.v4.f64 [%0], {%1, %2, %3, %4};" ::"l"(dst + k), "d"(z[k].x), "d"(z[k].y),
                         "d"(z[k + 1].x), "d"(z[k + 1].y) : "memory");
        } else {
            dst[k] = z[k];
            dst[k + 1] = z[k + 1];
        }
    }
}

__global__ void k_to_internal_f32(const double2* in, float2* __restrict__ out,
                                  int vol, int n) {
    pdl_enter();
    long t = blockIdx.x * (long)blockDim.x + threadIdx.x;
    if (t >= (long)vol * n) return;
    int r = (int)(t / vol), s = (int)(t % vol);
    const double2* src = in + ((size_t)r * vol + s) * 12;
    float2* dst = out + (size_t)r * 12 * vol;
    double2 z[12];
#pragma unroll
    for (int k = 0; k < 12; k++) z[k] = src[k];
#pragma unroll
    for (int k = 0; k < 12; k++) dst[sidx(k, s, vol)] = make_float2((float)z[k].x, (float)z[k].y);
}

__global__ void k_gauge_to_internal(const double2* __restrict__ in, double2* __restrict__ u64,
                                    float2* __restrict__ u32, int vol) {
    int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= vol) return;
    const double2* src = in + (size_t)s * 36;
#pragma unroll
    for (int e = 0; e < 36; e++) {  // e = mu*9 + 3a + b
        double2 z = src[e];
        u64[(size_t)e * vol + s] = z;
        u32[(size_t)e * vol + s] = make_float2((float)z.x, (float)z.y);
    }
}

// The result of field r at site s: internal planes, or the boundary's complex128 spinor, written in place of
// a separate widening pass (6 full 32-byte sectors per thread; 8^3 x 16, 12 fields: that pass took 8.2 us)
__device__ __forceinline__ void put_site(const OutF32& o, int r, int vol, int s, const Spinor<float>& v) {
    store_spinor(o.p + (size_t)r * 12 * vol, vol, s, v);
}
__device__ __forceinline__ void put_site(const OutF64& o, int r, int vol, int s, const Spinor<float>& v) {
    put_spinor_f64(o, (size_t)r * vol + s, v);
}

// ---------------------------------------------------------------------------
// one thread per site, field blockIdx.y, links and neighbours from global memory (coalesced:
// neighbouring threads read neighbouring sites).  PRE: the links are scaled before the product, as the tiles below
// have them, so that any number of fields gives the same bits.
// ---------------------------------------------------------------------------
template <int DAG, bool PRE, typename Out>
__global__ void __launch_bounds__(kThreads)
k_dslash(Geom g, const float2* __restrict__ u, float kappa, const float2* in, Out out) {
    pdl_enter();
    int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s >= g.vol) return;
    const int vol = g.vol;
    in += (size_t)blockIdx.y * 12 * vol;
    Nbr n = neighbours(g, s);
    Spinor<float> res;
    auto load = [&](int y, Spinor<float>& p) { load_spinor(in, vol, y, p); };
    if constexpr (PRE) {
        const float kf = n.fwrap_t ? kappa : -kappa, kb = n.bwrap_t ? kappa : -kappa;
        auto fl = [&](int mu, int e) {
            return cscale(__ldg(u + (size_t)(mu * 9 + e) * vol + s), mu == 3 ? kf : -kappa);
        };
        auto bl = [&](int mu, int e) {
            return cscale(__ldg(u + (size_t)(mu * 9 + e) * vol + n.b[mu]), mu == 3 ? kb : -kappa);
        };
        wilson_site_prescaled<DAG, float>(n, s, load, fl, bl, res);
    } else {
        auto fl = [&](int mu, int e) { return __ldg(u + (size_t)(mu * 9 + e) * vol + s); };
        auto bl = [&](int mu, int e) { return __ldg(u + (size_t)(mu * 9 + e) * vol + n.b[mu]); };
        wilson_site_ahead<DAG, 2>(n, s, load, fl, bl, kappa, res);
    }
    put_site(out, blockIdx.y, vol, s, res);
}

// ---------------------------------------------------------------------------
// multi right-hand side: a block owns 32 consecutive sites (a lane each) and all n fields, RPB warps side by
// side.  The 8 links of every site (U_mu(x) and U_mu(x-mu), times -kappa and the t-boundary sign) are staged
// once in shared memory.  The gathers' latency bounds it: many small blocks, a neighbour in flight per warp, the fields'
// plane addresses in uniform registers (see wilson_hops_prescaled and tile_blocks; D on 12 fields of 16^3 x 32 with
// a cold L2: 131 us with brick tiles of 64 sites at 80 registers and one gather in flight, 126 us here).
// ---------------------------------------------------------------------------
constexpr int TS = 32;

template <int DAG, int RPB, typename Out>
__global__ void __launch_bounds__(TS * RPB, tile_blocks(RPB))
k_dslash_mrhs(Geom g, const float2* __restrict__ u, float kappa, int n, const float2* in, Out out) {
    pdl_enter();
    __shared__ float2 sl[72 * TS];
    __shared__ OffNbr snb[TS];
    __shared__ int sb[4][TS];
    __shared__ float sgn[2][TS];
    const int vol = g.vol;
    const int s0 = blockIdx.x * TS;
    if (threadIdx.x < TS && s0 + threadIdx.x < vol) {
        const Nbr nb = neighbours(g, s0 + threadIdx.x);
        snb[threadIdx.x] = offsets_of(nb, 0);
#pragma unroll
        for (int mu = 0; mu < 4; mu++) sb[mu][threadIdx.x] = nb.b[mu];
        sgn[0][threadIdx.x] = nb.fwrap_t ? kappa : -kappa;
        sgn[1][threadIdx.x] = nb.bwrap_t ? kappa : -kappa;
    }
    __syncthreads();
    stage_tile_links<TS>(sl, u, vol, [&](int dir, int mu, int j, unsigned& site, float& scale) {
        if (s0 + j >= vol) return false;
        site = dir ? sb[mu][j] : s0 + j;
        scale = mu == 3 ? sgn[dir][j] : -kappa;
        return true;
    });
    __syncthreads();
    const int j = threadIdx.x % TS, s = s0 + j;
    const int q = uniform_warp(threadIdx.x / TS);
    if (s >= vol) return;
    const OffNbr& nb = snb[j];
    auto fl = [&](int mu, int e) { return sl[(mu * 9 + e) * TS + j]; };
    auto bl = [&](int mu, int e) { return sl[(36 + mu * 9 + e) * TS + j]; };
    const size_t plane = (size_t)vol * 16;
    for (int r = q; r < n; r += RPB) {
        links_stay_shared();
        const char* inr = reinterpret_cast<const char*>(in) + r * (6 * plane);
        Spinor<float> res;
        auto load = [&](unsigned o, Spinor<float>& p) { load_spinor_at(inr, plane, o, p); };
        wilson_site_prescaled<DAG, float>(nb, (unsigned)s * 16u, load, fl, bl, res);
        put_site(out, r, vol, s, res);
    }
}

template <int RPB, typename Out>
void mrhs_go(const Geom& g, const float2* u, float kappa, int dag, int n, const float2* in, Out out, cudaStream_t st) {
    const int nb = blocks_for(g.vol, TS);
    launch_pdl(pdl_for_apply(12L * g.vol * n), dag ? k_dslash_mrhs<1, RPB, Out> : k_dslash_mrhs<0, RPB, Out>, nb, TS * RPB,
               0, st, g, u, kappa, n, in, out);
}

template <bool PRE, typename Out>
void launch_dslash(const Geom& g, const float2* u, float kappa, int dag, int n, const float2* in, Out out,
                   cudaStream_t s) {
    // fields side by side in the grid
    for (int r0 = 0; r0 < n; r0 += kMaxGridY) {
        const dim3 grid(blocks_for(g.vol, kThreads), std::min(n - r0, kMaxGridY));
        const size_t off = (size_t)r0 * 12 * g.vol;
        Out o = out;
        if constexpr (std::is_same<Out, OutF64>::value) o.p += 2 * off;
        else o.p += off;
        launch_pdl(pdl_for_apply(12L * g.vol * (int)grid.y), dag ? k_dslash<1, PRE, Out> : k_dslash<0, PRE, Out>, grid, kThreads, 0, s,
                   g, u, kappa, in + off, o);
    }
}

// rpb warps per tile (0: the default); one or two fields have nothing to share a staged link with
template <typename Out>
void launch_dslash_mrhs(const Geom& g, const float2* u, float kappa, int dag, int n, const float2* in, Out out,
                        int rpb, cudaStream_t st) {
    if (n <= 2) {
        launch_dslash<true>(g, u, kappa, dag, n, in, out, st);
        return;
    }
    switch (rpb) {
        case 3: mrhs_go<3>(g, u, kappa, dag, n, in, out, st); break;
        case 6: mrhs_go<6>(g, u, kappa, dag, n, in, out, st); break;
        case 8: mrhs_go<8>(g, u, kappa, dag, n, in, out, st); break;
        case 12: mrhs_go<12>(g, u, kappa, dag, n, in, out, st); break;
        default: mrhs_go<4>(g, u, kappa, dag, n, in, out, st); break;
    }
}

// ---------------------------------------------------------------------------
// autotuner of the tile kernel: warps (fields side by side) per block, timed with CUDA events on the
// caller's own buffers at the first call for a (lattice, n, output, D or D^dag) and kept for the process (and in
// SEEDCG_TUNE_CACHE when set, as lines "brick_... warps 0 0").
// ---------------------------------------------------------------------------
template <typename Out>
int tuned_warps(const Geom& g, const float2* u, float kappa, int dag, int n, const float2* in, Out out,
                cudaStream_t st) {
    if (n <= 2) return 0;
    static std::mutex mu;
    static std::map<std::string, int> cache;
    char key[160];
    snprintf(key, sizeof(key), "brick_t32_%s_%dx%dx%dx%d_n%d_dag%d",
             std::is_same<Out, OutF64>::value ? "f32w" : "f32", g.L[0], g.L[1], g.L[2], g.L[3], n, dag);
    {
        std::lock_guard<std::mutex> lk(mu);
        auto it = cache.find(key);
        if (it != cache.end()) return it->second;
        if (const char* path = getenv("SEEDCG_TUNE_CACHE")) {
            FILE* f = fopen(path, "r");
            if (f) {
                // the file is shared with the batched-CG tuner: read only full lines of this one
                char line[640], k[512];
                int a, b, c;
                while (fgets(line, sizeof(line), f))
                    if (sscanf(line, "%511s %d %d %d", k, &a, &b, &c) == 4 && std::string(k) == key) cache[key] = a;
                fclose(f);
                it = cache.find(key);
                if (it != cache.end()) return it->second;
            }
        }
    }
    cudaStreamCaptureStatus cap_status = cudaStreamCaptureStatusNone;
    cudaStreamIsCapturing(st, &cap_status);
    if (cap_status != cudaStreamCaptureStatusNone) return 0;  // no timing inside a capture
    const bool tune_log = getenv("SEEDCG_TUNE_LOG") != nullptr;
    cudaEvent_t a, b;
    SEEDCG_CUDA_TRY(cudaEventCreate(&a));
    SEEDCG_CUDA_TRY(cudaEventCreate(&b));
    int best = 4;
    float best_ms = 1e30f;
    for (const int c : {3, 4, 6, 8, 12}) {
        if (c > 4 && c >= n + 3) continue;   // warps without a field
        launch_dslash_mrhs<Out>(g, u, kappa, dag, n, in, out, c, st);
        SEEDCG_CUDA_TRY(cudaEventRecord(a, st));
        for (int r = 0; r < 3; r++) launch_dslash_mrhs<Out>(g, u, kappa, dag, n, in, out, c, st);
        SEEDCG_CUDA_TRY(cudaEventRecord(b, st));
        SEEDCG_CUDA_TRY(cudaEventSynchronize(b));
        float ms = 0.f;
        SEEDCG_CUDA_TRY(cudaEventElapsedTime(&ms, a, b));
        if (tune_log) fprintf(stderr, "seedcg tune %s: %d warps: %.4f ms\n", key, c, ms / 3);
        if (ms < best_ms) {
            best_ms = ms;
            best = c;
        }
    }
    cudaEventDestroy(a);
    cudaEventDestroy(b);
    std::lock_guard<std::mutex> lk(mu);
    cache[key] = best;
    if (const char* path = getenv("SEEDCG_TUNE_CACHE")) {
        FILE* f = fopen(path, "a");
        if (f) {
            fprintf(f, "%s %d 0 0\n", key, best);
            fclose(f);
        }
    }
    return best;
}

}  // namespace

void to_internal_f64(const double* in, double2* out, int vol, int n, cudaStream_t s) {
    if ((long)vol * n == 0) return;
    k_to_internal_f64<<<blocks_for((long)vol * n, 256), 256, 0, s>>>(
        reinterpret_cast<const double2*>(in), out, vol, n);
    SEEDCG_CHECK_LAUNCH();
}
void from_internal_f64(const double2* in, double* out, int vol, int n, cudaStream_t s) {
    if ((long)vol * n == 0) return;
    k_from_internal_f64<<<blocks_for((long)vol * n, 256), 256, 0, s>>>(
        in, reinterpret_cast<double2*>(out), vol, n, (reinterpret_cast<uintptr_t>(out) & 31) == 0);
    SEEDCG_CHECK_LAUNCH();
}
void to_internal_f32(const double* in, float2* out, int vol, int n, cudaStream_t s) {
    if ((long)vol * n == 0) return;
    k_to_internal_f32<<<blocks_for((long)vol * n, 256), 256, 0, s>>>(
        reinterpret_cast<const double2*>(in), out, vol, n);
    SEEDCG_CHECK_LAUNCH();
}
void gauge_to_internal(const double* in, double2* u64, float2* u32, int vol, cudaStream_t s) {
    k_gauge_to_internal<<<blocks_for(vol, 256), 256, 0, s>>>(
        reinterpret_cast<const double2*>(in), u64, u32, vol);
    SEEDCG_CHECK_LAUNCH();
}

template <typename Out>
void dslash_mrhs_f32(const Geom& g, const float2* u, float kappa, int dag, int n, const float2* in, Out out,
                     bool fixed, cudaStream_t s) {
    if (n <= 0) return;
    launch_dslash_mrhs<Out>(g, u, kappa, dag, n, in, out, fixed ? 0 : tuned_warps<Out>(g, u, kappa, dag, n, in, out, s), s);
}
template void dslash_mrhs_f32<OutF32>(const Geom&, const float2*, float, int, int, const float2*, OutF32, bool, cudaStream_t);

void apply_spinors_f32(const Geom& g, const float2* u, float kappa, int op, int multi, bool fixed, int n,
                       const double* in, double* out, float2* work, cudaStream_t s) {
    to_internal_f32(in, work, g.vol, n, s);
    auto go = [&](int dag, const float2* x, auto y) {
        if (multi) dslash_mrhs_f32(g, u, kappa, dag, n, x, y, fixed, s);
        else launch_dslash<false>(g, u, kappa, dag, n, x, y, s);
    };
    float2* t = work + (size_t)n * 12 * g.vol;
    if (op < 2) {
        go(op, work, make_out_f64(out));
    } else {
        go(0, work, OutF32{t});
        go(1, t, make_out_f64(out));
    }
}
}  // namespace seedcg
