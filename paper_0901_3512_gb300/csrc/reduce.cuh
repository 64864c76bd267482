// Deterministic block and grid reductions in FP64.
//
// Every reducing kernel writes one partial per block into a fixed slot; the
// last block to finish (elected through an atomic ticket) sums the slots in
// a fixed order and runs the finalisation on one thread.  The result does not
// depend on block scheduling, so repeated runs are bitwise identical.
#pragma once

#include "grids.h"
#include "internal.cuh"

namespace seedcg {

// warp sum in the value's own precision (FP32 sums stay off the scarce FP64 pipe)
template <typename T> __device__ __forceinline__ T warp_sum_t(T v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    return v;
}

// float -> double by moving bits: the conversion instruction is on the FP64 pipe, which takes 68 clocks per warp
__device__ __forceinline__ double widen(float x) {
    const unsigned b = __float_as_uint(x), m = b & 0x7fffffffu;
    const bool normal = m - 0x00800000u < 0x7f000000u;
    if (!normal && m != 0u) return (double)x;   // subnormal, infinite or NaN
    return __hiloint2double((int)((b & 0x80000000u) | (normal ? (m >> 3) + 0x38000000u : 0u)), (int)(b << 29));
}
__device__ __forceinline__ double widen(double x) { return x; }
// and back, rounded to nearest even
__device__ __forceinline__ float narrow(double x) {
    const long long b = __double_as_longlong(x);
    const unsigned long long u = (unsigned long long)b & 0x7fffffffffffffffull;
    const unsigned e = (unsigned)(u >> 52);
    if (u != 0 && e - 897u >= 254u) return (float)x;   // outside FP32's normal range, infinite or NaN
    const unsigned long long v = u - (896ull << 52);
    const unsigned r = (unsigned)((v + 0x0fffffffull + ((v >> 29) & 1u)) >> 29);
    return __uint_as_float((u == 0 ? 0u : r) | ((unsigned)((unsigned long long)b >> 32) & 0x80000000u));
}
// 1 / x rounded once: FP32 in two floats (x = h + l), as an FP64 division by every thread holds its pipe for 1 us per
// block.  Far from 1 the scaling of l would leave FP32's range: the FP64 division.
template <typename R> __device__ __forceinline__ R inverse(double x) {
    if constexpr (sizeof(R) == 8) {
        return 1.0 / x;
    } else {
        const unsigned long long b = (unsigned long long)__double_as_longlong(x);
        const unsigned e = (unsigned)(b >> 52);
        if (e - 960u >= 128u) return (float)(1.0 / x);   // also negative, infinite or NaN
        const float h = __uint_as_float((unsigned)((b - (896ull << 52)) >> 29));
        const float l = (float)(unsigned)(b & 0x1fffffffu) * __uint_as_float((e - 948u) << 23);
        const float r = 1.f / h;
        return fmaf(r, fmaf(-l, r, fmaf(-h, r, 1.f)), r);
    }
}
template <typename R> __device__ __forceinline__ R to_real(double x) {
    if constexpr (sizeof(R) == 4) return narrow(x);
    else return x;
}

// Sum over a warp, on every lane. Five shuffled FP64 additions are about 900 clocks in a row, and four warps of a
// partition take turns on its pipe; so the lanes' values are taken as integers relative to the largest exponent E
// (58 bits, the lowest one rounded), added exactly by the warp's integer reductions in three parts and rounded once:
// about 600 clocks, which warps overlap, and an error of at most 2^-53 of the largest value and of the sum against 5 * 2^-53 of the partial sums. Values next to the ends of
// FP64's range, infinities and NaN take the additions.
__device__ __forceinline__ double warp_sum(double v) {
    const int hi = __double2hiint(v), e = (hi >> 20) & 0x7ff;
    const int E = (int)__reduce_max_sync(0xffffffffu, (unsigned)e);
    if (E < 64 || E > 2040) {
        if (E == 0 && __all_sync(0xffffffffu, v == 0.0)) return 0.0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        return v;
    }
    const unsigned long long mant = ((unsigned long long)(unsigned)((hi & 0xfffff) | 0x100000) << 32) | (unsigned)__double2loint(v);
    const int d = E - e;
    const unsigned long long t = e == 0 ? 0ull : mant << 5;   // a subnormal is below 2^-62 of the largest
    const unsigned long long r = d == 0 ? t : ((t >> (d < 64 ? d - 1 : 63)) + 1) >> 1;
    const long long q = hi < 0 ? -(long long)r : (long long)r;
    const unsigned s0 = __reduce_add_sync(0xffffffffu, (unsigned)q & 0x7ffffffu);
    const unsigned s1 = __reduce_add_sync(0xffffffffu, (unsigned)(q >> 27) & 0x7ffffffu);
    const int s2 = __reduce_add_sync(0xffffffffu, (int)(q >> 54));
    const long long sum = (long long)(((unsigned long long)(long long)s2 << 54) + ((unsigned long long)s1 << 27) + s0);
    if (sum == 0) return 0.0;
    const double x = (double)sum;   // 2^(E - 1080) too large; every exponent on the way is a normal one
    return __hiloint2double(__double2hiint(x) + ((E - 1080) << 20), __double2loint(x));
}

// the warps' sums of one value (at most four: three additions are shorter than a warp_sum), in a fixed tree
__device__ __forceinline__ double sum_warps(const double* w, int nw) {
    double t = w[0];
    if (nw > 1) t += w[1];
    if (nw > 2) t += nw > 3 ? w[2] + w[3] : w[2];
    return t;
}
template <int NV>
__device__ __forceinline__ void warp_sums(const double (&v)[NV], double (&sh)[NV][kRedThreads / 32]) {
#pragma unroll
    for (int k = 0; k < NV; k++) {
        const double t = warp_sum(v[k]);
        if ((threadIdx.x & 31) == 0) sh[k][threadIdx.x >> 5] = t;
    }
    __syncthreads();
}

// Sum v[k] over the block (at most kRedThreads threads); the first warp holds the totals. Two calls need a barrier between.
template <int NV>
__device__ __forceinline__ void block_sum(double (&v)[NV]) {
    static_assert(NV <= 32, "one lane per value");
    __shared__ double sh[NV][kRedThreads / 32];
    warp_sums<NV>(v, sh);
    if (threadIdx.x >= 32) return;
    const int nw = (blockDim.x + 31) >> 5;
    if (nw > 4) {
#pragma unroll
        for (int k = 0; k < NV; k++) v[k] = warp_sum((int)threadIdx.x < nw ? sh[k][threadIdx.x] : 0.0);
        return;
    }
    const double t = threadIdx.x < NV ? sum_warps(sh[threadIdx.x], nw) : 0.0;
#pragma unroll
    for (int k = 0; k < NV; k++) v[k] = NV == 1 ? t : __shfl_sync(0xffffffffu, t, k);
}
// the same for more values, held by every thread
template <int NV>
__device__ __forceinline__ void block_sum_all(double (&v)[NV]) {
    __shared__ double sh[NV][kRedThreads / 32];
    warp_sums<NV>(v, sh);
    for (int k = threadIdx.x; k < NV; k += blockDim.x) {
        double t = sh[k][0];
        for (int w = 1; w < (int)(blockDim.x + 31) >> 5; w++) t += sh[k][w];
        sh[k][0] = t;
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < NV; k++) v[k] = sh[k][0];
}

// Grid-wide sum over a 1-D or 2-D grid.  partials holds NV * nblocks doubles,
// counter one unsigned that is zero on entry (it is reset on exit).  fin(tot, pre)
// runs once, on thread 0 of the last block, with the grid totals; aux(pre) is what
// does not need them, done by another warp of that block meanwhile: scalar work (an
// FP64 division is about 900 clocks here) and the loads that fin would wait for (each
// about 600), up to kAuxValues results in shared memory.
constexpr int kAuxValues = 6;
template <int NV, typename Aux, typename Fin>
__device__ __forceinline__ void grid_sum(double (&v)[NV], double* partials, unsigned* counter,
                                         Aux aux, Fin fin) {
    __shared__ bool s_last;
    __shared__ double s_pre[kAuxValues];
    block_sum<NV>(v);
    const unsigned nblk = gridDim.x * gridDim.y;
    const unsigned bid = blockIdx.y * gridDim.x + blockIdx.x;
    if (threadIdx.x == 0) {
#pragma unroll
        for (int k = 0; k < NV; k++) partials[(size_t)k * nblk + bid] = v[k];
        // one ordered ticket: the block's partials before it, the other blocks' after (for the block, by the barrier)
        unsigned t;
        asm volatile("atom.add.acq_rel.gpu.global.u32 %0, [%1], 1;" : "=r"(t) : "l"(counter) : "memory");
        s_last = (t == nblk - 1);
    }
    __syncthreads();
    if (!s_last) return;
    if (threadIdx.x == blockDim.x - 1) {
        aux(s_pre);
        *counter = 0u;   // every block has drawn its ticket; the next kernel sees it
    }
    double tot[NV];
#pragma unroll
    for (int k = 0; k < NV; k++) tot[k] = 0.0;
    // the loads of up to eight partials before their additions; few partials are left to one warp
    constexpr int U = NV <= 2 ? 8 : 1;
    const unsigned bd = nblk <= 128 ? 32 : blockDim.x;
    if (threadIdx.x < bd) {
        for (unsigned b0 = 0; b0 < nblk; b0 += U * bd) {
            double p[U][NV];
#pragma unroll
            for (int u = 0; u < U; u++) {
                const unsigned b = b0 + u * bd + threadIdx.x;
#pragma unroll
                for (int k = 0; k < NV; k++) p[u][k] = b < nblk ? __ldcg(partials + (size_t)k * nblk + b) : 0.0;
            }
#pragma unroll
            for (int u = 0; u < U; u++)
                if (b0 + u * bd < nblk)
#pragma unroll
                    for (int k = 0; k < NV; k++) tot[k] += p[u][k];
        }
    }
    if (nblk <= 128) {
        if (threadIdx.x < 32)
#pragma unroll
            for (int k = 0; k < NV; k++) tot[k] = warp_sum(tot[k]);
        __syncthreads();   // aux is done
    } else {
        block_sum<NV>(tot);
    }
    if (threadIdx.x == 0) fin(tot, s_pre);
}
template <int NV, typename Fin>
__device__ __forceinline__ void grid_sum(double (&v)[NV], double* partials, unsigned* counter,
                                         Fin fin) {
    grid_sum<NV>(v, partials, counter, [](double*) {}, [&](double* tot, const double*) { fin(tot); });
}

// ---------------------------------------------------------------------------
// loads of one complex entry from the three storage types, widened to R
// ---------------------------------------------------------------------------
template <typename R> __device__ __forceinline__ cx_t<R> ld_cx(const double2* p, size_t i) {
    double2 z = p[i]; return mk<R>((R)z.x, (R)z.y);
}
template <typename R> __device__ __forceinline__ cx_t<R> ld_cx(const float2* p, size_t i) {
    float2 z = p[i]; return mk<R>((R)z.x, (R)z.y);
}
template <typename R> __device__ __forceinline__ cx_t<R> ld_cx(const __nv_bfloat162* p, size_t i) {
    float2 z = __bfloat1622float2(p[i]); return mk<R>((R)z.x, (R)z.y);
}
__device__ __forceinline__ void st_cx(double2* p, size_t i, double2 z) { p[i] = z; }
__device__ __forceinline__ void st_cx(double2* p, size_t i, float2 z) { p[i] = make_double2(z.x, z.y); }
__device__ __forceinline__ void st_cx(float2* p, size_t i, double2 z) { p[i] = make_float2((float)z.x, (float)z.y); }
__device__ __forceinline__ void st_cx(float2* p, size_t i, float2 z) { p[i] = z; }
__device__ __forceinline__ void st_cx(__nv_bfloat162* p, size_t i, float2 z) { p[i] = __float22bfloat162_rn(z); }
__device__ __forceinline__ void st_cx(__nv_bfloat162* p, size_t i, double2 z) {
    p[i] = __float22bfloat162_rn(make_float2((float)z.x, (float)z.y));
}

// One 16-byte load of consecutive complex elements of type VT (1 double2,
// 2 float2 or 4 bf16x2), widened to cx_t<R>; marked streaming (evict-first):
// the stored basis is read once per use and should not push the iteration
// vectors out of L2.  p must be 16-byte aligned.
template <typename R, typename VT> struct VLoad;
template <typename R> struct VLoad<R, double2> {
    static constexpr int N = 1;
    __device__ __forceinline__ static void get(const double2* p, cx_t<R> (&o)[1]) {
        const double2 z = __ldcs(p);
        o[0] = mk<R>((R)z.x, (R)z.y);
    }
};
template <typename R> struct VLoad<R, float2> {
    static constexpr int N = 2;
    __device__ __forceinline__ static void get(const float2* p, cx_t<R> (&o)[2]) {
        const float4 z = __ldcs(reinterpret_cast<const float4*>(p));
        o[0] = mk<R>((R)z.x, (R)z.y);
        o[1] = mk<R>((R)z.z, (R)z.w);
    }
};
template <typename R> struct VLoad<R, __nv_bfloat162> {
    static constexpr int N = 4;
    __device__ __forceinline__ static void get(const __nv_bfloat162* p, cx_t<R> (&o)[4]) {
        const uint4 z = __ldcs(reinterpret_cast<const uint4*>(p));
        const unsigned w[4] = {z.x, z.y, z.z, z.w};
#pragma unroll
        for (int k = 0; k < 4; k++) {
            __nv_bfloat162 b;
            memcpy(&b, &w[k], 4);
            const float2 f = __bfloat1622float2(b);
            o[k] = mk<R>((R)f.x, (R)f.y);
        }
    }
};

}  // namespace seedcg
