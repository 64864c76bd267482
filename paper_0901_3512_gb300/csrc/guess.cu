// Learned initial guess: a gauge-covariant nearest-neighbour network
//   out_co(x) = sum_ci [ W_0[co,ci] in_ci(x) + sum_{d=+-mu} W_d[co,ci] U(x,d) in_ci(x+d) ]
// (U(x,+mu) = U_mu(x), U(x,-mu) = U_mu(x-mu)^dag, antiperiodic-t sign as in D;
// W_d[co,ci] a complex 4x4 spin matrix; channels 1 -> 8 -> 8 -> 1; ReLU on real
// and imaginary parts after layers 1 and 2; input b/||b||, output times ||b||),
// with hand-written forward, backward and Adam kernels.
//
// Storage is bf16, accumulation FP32: activations, their gradients and the
// weights the layers read are bf16; Adam keeps an FP32 master copy of the
// weights and FP32 moments, and the weight gradient is summed in FP64.
//
// Layer 2 (8 -> 8) is a dense contraction with K = 9 directions x 8 channels x 4
// spins = 288 complex terms per output, run on the tcgen05 tensor cores as the
// real GEMM  D[site][n] = sum_k A[site][k] B[n][k]  per colour:
//   A = the link-transported neighbour activations of 128 sites (built by the CTA
//       in shared memory, one direction d per 64-wide K chunk),
//   B = the layer's weights in real form (64 x 64 bf16 per direction),
//   D = 128 x 64 FP32 accumulators in TMEM, one per colour.
// The backward pass through the data of layer 2 is the same GEMM with the
// adjoint transport and the adjoint weights, and the weight gradients of all layers run on
// tcgen05 too (k_g_tw).  Layers 1 and 3 (one channel on one side) run on SIMT.
//
// Activations are bf16x2 [C][V][12] (entry k = 3 spin + colour of site x at
// (c V + x) 12 + k); weights of a layer are [9][CO][CI][4][4] complex, directions
// 0 (on site), +x,-x,+y,-y,+z,-z,+t,-t.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include "handle.cuh"
#include "kernels.cuh"
#include "reduce.cuh"
#include "tc_common.cuh"
#include "wilson.cuh"

namespace seedcg {

namespace {

using bf2 = __nv_bfloat162;

// ---------------------------------------------------------------------------
// bf16 site records: the 12 complex entries of one channel at one site, 48 bytes
// ---------------------------------------------------------------------------
__device__ __forceinline__ float2 unpack_bf2(unsigned w) {
    bf2 b;
    memcpy(&b, &w, 4);
    return __bfloat1622float2(b);
}
__device__ __forceinline__ unsigned pack_bf2(float2 v) {
    const bf2 b = __float22bfloat162_rn(v);
    unsigned w;
    memcpy(&w, &b, 4);
    return w;
}
__device__ __forceinline__ void ld_site(const bf2* __restrict__ p, float2 (&o)[12]) {
    const uint4* q = reinterpret_cast<const uint4*>(p);
#pragma unroll
    for (int j = 0; j < 3; j++) {
        const uint4 a = __ldg(q + j);
        o[4 * j + 0] = unpack_bf2(a.x);
        o[4 * j + 1] = unpack_bf2(a.y);
        o[4 * j + 2] = unpack_bf2(a.z);
        o[4 * j + 3] = unpack_bf2(a.w);
    }
}
__device__ __forceinline__ void st_site(bf2* __restrict__ p, const float2 (&v)[12]) {
    uint4* q = reinterpret_cast<uint4*>(p);
#pragma unroll
    for (int j = 0; j < 3; j++)
        q[j] = make_uint4(pack_bf2(v[4 * j]), pack_bf2(v[4 * j + 1]), pack_bf2(v[4 * j + 2]), pack_bf2(v[4 * j + 3]));
}
__device__ __forceinline__ const bf2* site_ptr(const bf2* a, int ch, int vol, int x) {
    return a + ((size_t)ch * vol + x) * 12;
}
__device__ __forceinline__ bf2* site_ptr(bf2* a, int ch, int vol, int x) {
    return a + ((size_t)ch * vol + x) * 12;
}

// Where direction d's term at site x comes from: the activation of site src, carried by the link at site
// lsite in direction mu (its adjoint when dag), times sg.  ADJ: the adjoint transport of the backward pass
// through the data (the hop from src in direction d, seen from x).
struct HopFrom {
    int src, lsite, mu;
    bool dag;
    float sg;
};
template <bool ADJ>
__device__ __forceinline__ HopFrom hop_from(const Geom& g, int x, int d) {
    HopFrom h{x, x, 0, false, 1.f};
    if (d == 0) return h;
    h.mu = (d - 1) >> 1;
    const bool back = ((d - 1) & 1) != (ADJ ? 1 : 0);   // src = x - mu
    const int str = h.mu == 0 ? g.stride[0] : h.mu == 1 ? g.stride[1] : h.mu == 2 ? g.stride[2] : g.stride[3];
    const int ext = h.mu == 0 ? g.L[0] : h.mu == 1 ? g.L[1] : h.mu == 2 ? g.L[2] : g.L[3];
    const int c = (x / str) % ext;
    const bool wrap = back ? c == 0 : c == ext - 1;
    h.src = back ? (wrap ? x + (ext - 1) * str : x - str) : (wrap ? x - (ext - 1) * str : x + str);
    h.lsite = back ? h.src : x;
    h.dag = back;
    h.sg = h.mu == 3 && wrap ? -1.f : 1.f;
    return h;
}

// One thread's loads for a direction, issued ahead of their use: the link and NCH channels of the source site
template <int NCH>
struct HopLoad {
    float2 lk[9];
    uint4 act[NCH][3];
    bool dag;
    float sg;
};
template <bool ADJ, int NCH>
__device__ __forceinline__ void hop_load(HopLoad<NCH>& p, const Geom& g, const float2* __restrict__ u,
                                         const bf2* __restrict__ in, int ch0, int x, int d) {
    const HopFrom h = hop_from<ADJ>(g, x, d);
    p.dag = h.dag;
    p.sg = h.sg;
#pragma unroll
    for (int k = 0; k < NCH; k++) {
        const uint4* q = reinterpret_cast<const uint4*>(site_ptr(in, ch0 + k, g.vol, h.src));
#pragma unroll
        for (int j = 0; j < 3; j++) p.act[k][j] = __ldg(q + j);
    }
    if (d > 0) {
        const float2* l = u + (size_t)(h.mu * 9) * g.vol + h.lsite;
#pragma unroll
        for (int e = 0; e < 9; e++) p.lk[e] = __ldg(l + (size_t)e * g.vol);
    }
}
// the link as the matrix that transports colour vectors (sign and adjoint applied)
template <int NCH>
__device__ __forceinline__ void hop_matrix(const HopLoad<NCH>& p, float2 (&m)[9]) {
#pragma unroll
    for (int a = 0; a < 3; a++)
#pragma unroll
        for (int b = 0; b < 3; b++) {
            const float2 z = p.dag ? p.lk[3 * b + a] : p.lk[3 * a + b];
            m[3 * a + b] = make_float2(p.sg * z.x, p.dag ? -p.sg * z.y : p.sg * z.y);
        }
}
__device__ __forceinline__ void unpack_site(const uint4 (&w)[3], float2 (&o)[12]) {
#pragma unroll
    for (int j = 0; j < 3; j++) {
        o[4 * j + 0] = unpack_bf2(w[j].x);
        o[4 * j + 1] = unpack_bf2(w[j].y);
        o[4 * j + 2] = unpack_bf2(w[j].z);
        o[4 * j + 3] = unpack_bf2(w[j].w);
    }
}

// o = m v
__device__ __forceinline__ void colour_mul(const float2 (&m)[9], const float2* v, float2* o) {
#pragma unroll
    for (int a = 0; a < 3; a++) {
        float2 acc = make_float2(0.f, 0.f);
#pragma unroll
        for (int b = 0; b < 3; b++) acc = cfma(m[3 * a + b], v[b], acc);
        o[a] = acc;
    }
}

// ---------------------------------------------------------------------------
// SIMT layers (one channel on one side).  A block owns 32 sites (a lane each); every transported
// activation is formed once per (site, direction, channel) and shared through shared memory, where
// one thread per (site, output channel) formed it anew for each output before.  The sums keep the order
// direction, input channel, input spin, so the results are those of one thread running the whole chain.
// ---------------------------------------------------------------------------
constexpr int SL = 32;   // sites per block

// links of the block's sites in the eight directions, times the boundary sign: U(x,d) (ADJ = false) or the
// link that carries direction d's contribution back to x (apply_link_adj); sl[(d - 1) * 9 + e][lane]
template <bool ADJ>
__device__ __forceinline__ void stage_links(const Geom& gm, const float2* __restrict__ u, int x0,
                                            float2 (*sl)[SL], int (*snb)[SL]) {
    const int vol = gm.vol;
    for (int t = threadIdx.x; t < 8 * SL; t += blockDim.x) {
        const int j = t % SL, d = 1 + t / SL, x = x0 + j;
        if (x >= vol) continue;
        const Nbr nb = neighbours(gm, x);
        const int mu = (d - 1) >> 1;
        const bool back = (d - 1) & 1;
        // ADJ: direction +mu comes from x - mu over U_mu(x - mu)^dag, direction -mu from x + mu over U_mu(x)
        const bool src_back = ADJ ? !back : back;
        const int y = src_back ? nb.b[mu] : nb.f[mu];
        const int site = src_back ? y : x;
        const float sg = (mu == 3 && (src_back ? nb.bwrap_t : nb.fwrap_t)) ? -1.f : 1.f;
        snb[d - 1][j] = y;
#pragma unroll
        for (int e = 0; e < 9; e++) {
            const float2 z = __ldg(u + (size_t)(mu * 9 + e) * vol + site);
            sl[(d - 1) * 9 + e][j] = make_float2(sg * z.x, sg * z.y);
        }
    }
}

// the matrix that transports colour vectors, in registers: L or L^dag with L[a][b] = sl[3 a + b][lane]
__device__ __forceinline__ void staged_link(const float2 (*sl)[SL], int lane, bool dag, float2 (&m)[9]) {
#pragma unroll
    for (int a = 0; a < 3; a++)
#pragma unroll
        for (int b = 0; b < 3; b++) {
            const float2 z = sl[dag ? 3 * b + a : 3 * a + b][lane];
            m[3 * a + b] = make_float2(z.x, dag ? -z.y : z.y);
        }
}

// g_d(x) of one channel into sg[12][lane], in two parts: the source site's values on their way, and the rest
__device__ __forceinline__ void gather_load(const bf2* __restrict__ in_ch, int x, int d, const int (*snb)[SL], int lane,
                                            uint4 (&q)[3]) {
    const uint4* p = reinterpret_cast<const uint4*>(in_ch + (size_t)(d == 0 ? x : snb[d - 1][lane]) * 12);
#pragma unroll
    for (int j = 0; j < 3; j++) q[j] = __ldg(p + j);
}
__device__ __forceinline__ void gather_put(const uint4 (&q)[3], int d, const float2 (*sl)[SL], int lane,
                                           float2 (*sg)[SL]) {
    float2 v[12];
#pragma unroll
    for (int j = 0; j < 3; j++) {
        v[4 * j + 0] = unpack_bf2(q[j].x);
        v[4 * j + 1] = unpack_bf2(q[j].y);
        v[4 * j + 2] = unpack_bf2(q[j].z);
        v[4 * j + 3] = unpack_bf2(q[j].w);
    }
    if (d == 0) {
#pragma unroll
        for (int k = 0; k < 12; k++) sg[k][lane] = v[k];
        return;
    }
    float2 m[9], o[12];
    staged_link(sl + (d - 1) * 9, lane, (d - 1) & 1, m);
#pragma unroll
    for (int s = 0; s < 4; s++) colour_mul(m, &v[3 * s], &o[3 * s]);
#pragma unroll
    for (int k = 0; k < 12; k++) sg[k][lane] = o[k];
}

__device__ __forceinline__ void load_w(const bf2* __restrict__ w, float2 (&o)[16]) {
    const uint4* q = reinterpret_cast<const uint4*>(w);
#pragma unroll
    for (int j = 0; j < 4; j++) {
        const uint4 a = __ldg(q + j);
        o[4 * j + 0] = unpack_bf2(a.x);
        o[4 * j + 1] = unpack_bf2(a.y);
        o[4 * j + 2] = unpack_bf2(a.z);
        o[4 * j + 3] = unpack_bf2(a.w);
    }
}

// layer 1 (1 -> 8): nine warps transport one direction each, then eight warps run one output channel each.
// z may be null (inference needs h = ReLU(z) only).  16^3 x 32: 294 us with a thread per (site, output
// channel), 108 us here.
__global__ void __launch_bounds__(288)
k_g_first(Geom gm, const float2* __restrict__ u, const bf2* __restrict__ W, const bf2* __restrict__ in,
          bf2* __restrict__ z, bf2* __restrict__ h) {
    __shared__ float2 sl[72][SL];
    __shared__ int snb[8][SL];
    __shared__ float2 sg[9 * 12][SL];
    const int vol = gm.vol, x0 = blockIdx.x * SL;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, x = x0 + lane;
    const bool live = x < vol;
    stage_links<false>(gm, u, x0, sl, snb);
    __syncthreads();
    if (live) {
        uint4 q[3];
        gather_load(in, x, warp, snb, lane, q);
        gather_put(q, warp, sl, lane, sg + 12 * warp);
    }
    __syncthreads();
    if (warp >= 8 || !live) return;
    float2 acc[4][3];
#pragma unroll
    for (int k = 0; k < 12; k++) acc[k / 3][k % 3] = make_float2(0.f, 0.f);
#pragma unroll 1
    for (int d = 0; d < 9; d++) {
        float2 w[16], g[12];
        load_w(W + ((size_t)d * 8 + warp) * 16, w);
#pragma unroll
        for (int k = 0; k < 12; k++) g[k] = sg[12 * d + k][lane];
#pragma unroll
        for (int s = 0; s < 4; s++)
#pragma unroll
            for (int sp = 0; sp < 4; sp++)
#pragma unroll
                for (int c = 0; c < 3; c++) acc[s][c] = cfma(w[4 * s + sp], g[3 * sp + c], acc[s][c]);
    }
    float2 v[12], r[12];
#pragma unroll
    for (int k = 0; k < 12; k++) {
        v[k] = acc[k / 3][k % 3];
        r[k] = make_float2(fmaxf(v[k].x, 0.f), fmaxf(v[k].y, 0.f));
    }
    if (z) st_site(site_ptr(z, warp, vol, x), v);
    st_site(site_ptr(h, warp, vol, x), r);
}

// layer 3 (8 -> 1): eight warps transport one input channel each for direction d + 1 while three warps add
// direction d, a colour's four spins each, over the eight channels; the buffer of a direction is reused two later.
// Shared memory bounds it (two wavefronts per value read): with four spins per value instead of two 16^3 x 32 takes
// 190 us instead of 214 (346 with one thread per site); a producer loads a direction ahead.
constexpr int kLastThreads = 352;
__global__ void __launch_bounds__(kLastThreads, 2)
k_g_last(Geom gm, const float2* __restrict__ u, const bf2* __restrict__ W, const bf2* __restrict__ in,
         bf2* __restrict__ z) {
    extern __shared__ __align__(16) unsigned char last_smem[];
    float2 (*sl)[SL] = reinterpret_cast<float2 (*)[SL]>(last_smem);                        // [72]
    float2 (*sg)[SL] = sl + 72;                                                            // [2][8 * 12]
    float2 (*sw)[16] = reinterpret_cast<float2 (*)[16]>(sg + 2 * 96);                      // [9 * 8] weights
    int (*snb)[SL] = reinterpret_cast<int (*)[SL]>(sw + 72);                               // [8]
    bf2 (*so)[12] = reinterpret_cast<bf2 (*)[12]>(snb + 8);                                // [SL] results
    const int vol = gm.vol, x0 = blockIdx.x * SL;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, x = x0 + lane;
    const bool live = x < vol;
    stage_links<false>(gm, u, x0, sl, snb);
    // weights [d][ci][input spin][output spin]: two 16-byte loads give the four output spins
    for (int t = threadIdx.x; t < 72 * 16; t += blockDim.x)
        sw[t / 16][(t % 4) * 4 + (t / 4) % 4] = __bfloat1622float2(W[t]);
    __syncthreads();
    const bool producer = warp < 8;
    const bf2* in_ch = in + (size_t)warp * vol * 12;   // (producers)
    uint4 raw[3];
    if (producer && live) {
        gather_load(in_ch, x, 0, snb, lane, raw);
        gather_put(raw, 0, sl, lane, sg + 12 * warp);
        gather_load(in_ch, x, 1, snb, lane, raw);
    }
    const int c = warp - 8;   // consumer: colour c
    float2 acc[4];
#pragma unroll
    for (int s = 0; s < 4; s++) acc[s] = make_float2(0.f, 0.f);
#pragma unroll 1
    for (int d = 0; d < 9; d++) {
        __syncthreads();
        if (producer) {
            if (d < 8 && live) {
                gather_put(raw, d + 1, sl, lane, sg + ((d + 1) & 1) * 96 + 12 * warp);
                if (d < 7) gather_load(in_ch, x, d + 2, snb, lane, raw);
            }
        } else {
            const float2 (*g)[SL] = sg + (d & 1) * 96;
#pragma unroll
            for (int ci = 0; ci < 8; ci++) {
                const float2* w = sw[d * 8 + ci];
#pragma unroll
                for (int sp = 0; sp < 4; sp++) {
                    const float2 gv = g[12 * ci + 3 * sp + c][lane];
                    const float4 w0 = *reinterpret_cast<const float4*>(w + 4 * sp);
                    const float4 w1 = *reinterpret_cast<const float4*>(w + 4 * sp + 2);
                    acc[0] = cfma(make_float2(w0.x, w0.y), gv, acc[0]);
                    acc[1] = cfma(make_float2(w0.z, w0.w), gv, acc[1]);
                    acc[2] = cfma(make_float2(w1.x, w1.y), gv, acc[2]);
                    acc[3] = cfma(make_float2(w1.z, w1.w), gv, acc[3]);
                }
            }
        }
    }
    if (!producer) {
#pragma unroll
        for (int s = 0; s < 4; s++) so[lane][3 * s + c] = __float22bfloat162_rn(acc[s]);
    }
    __syncthreads();
    // the block's results are contiguous in z: [site][12]
    const int cnt = min(SL, vol - x0) * 12;
    for (int t = threadIdx.x; t < cnt; t += blockDim.x) z[(size_t)x0 * 12 + t] = so[t / 12][t % 12];
}

constexpr size_t kLastSmem = (72 + 2 * 96) * SL * sizeof(float2) + 72 * 16 * sizeof(float2) + 8 * SL * sizeof(int) +
                             SL * 12 * sizeof(bf2);

// backward through the data of layer 3: din[ci](y) = sum_d adjoint transport of W_d^dag dout (a warp per ci),
// times the ReLU mask of zprev; links and the neighbours' dout come from shared memory.  16^3 x 32: 410 -> 188 us.
__global__ void __launch_bounds__(256)
k_g_bwd_data(Geom gm, const float2* __restrict__ u, const bf2* __restrict__ W, const bf2* __restrict__ dout,
             const bf2* __restrict__ zprev, bf2* __restrict__ din) {
    __shared__ float2 sl[72][SL];
    __shared__ int snb[8][SL];
    __shared__ float2 sd[3][12][SL];   // dout of direction d at d % 3
    const int vol = gm.vol, y0 = blockIdx.x * SL;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, y = y0 + lane;
    const bool live = y < vol;
    stage_links<true>(gm, u, y0, sl, snb);
    __syncthreads();
    // the warps take turns to widen a direction's dout, two directions ahead
    auto fetch = [&](int d) {
        if (warp == d % 8 && live) {
            float2 v[12];
            ld_site(dout + (size_t)(d == 0 ? y : snb[d - 1][lane]) * 12, v);
#pragma unroll
            for (int k = 0; k < 12; k++) sd[d % 3][k][lane] = v[k];
        }
    };
    fetch(0);
    fetch(1);
    float2 acc[4][3];
#pragma unroll
    for (int k = 0; k < 12; k++) acc[k / 3][k % 3] = make_float2(0.f, 0.f);
#pragma unroll 1
    for (int d = 0; d < 9; d++) {
        __syncthreads();
        if (d + 2 < 9) fetch(d + 2);
        if (!live) continue;
        float2 w[16], dg[4][3];
        load_w(W + ((size_t)d * 8 + warp) * 16, w);
#pragma unroll
        for (int k = 0; k < 12; k++) dg[k / 3][k % 3] = make_float2(0.f, 0.f);
#pragma unroll
        for (int s = 0; s < 4; s++)
#pragma unroll
            for (int c = 0; c < 3; c++) {
                const float2 dv = sd[d % 3][3 * s + c][lane];
#pragma unroll
                for (int sp = 0; sp < 4; sp++) dg[sp][c] = cfma_conj(w[4 * s + sp], dv, dg[sp][c]);
            }
        if (d == 0) {
#pragma unroll
            for (int k = 0; k < 12; k++) acc[k / 3][k % 3] = cadd(acc[k / 3][k % 3], dg[k / 3][k % 3]);
        } else {
            float2 m[9];
            staged_link(sl + (d - 1) * 9, lane, d & 1, m);   // direction +mu (odd d) comes back over the adjoint
#pragma unroll
            for (int s = 0; s < 4; s++) {
                float2 o[3];
                colour_mul(m, dg[s], o);
#pragma unroll
                for (int c = 0; c < 3; c++) acc[s][c] = cadd(acc[s][c], o[c]);
            }
        }
    }
    if (!live) return;
    float2 v[12], zz[12];
    ld_site(site_ptr(zprev, warp, vol, y), zz);
#pragma unroll
    for (int k = 0; k < 12; k++) {
        const float2 a = acc[k / 3][k % 3];
        v[k] = make_float2(zz[k].x > 0.f ? a.x : 0.f, zz[k].y > 0.f ? a.y : 0.f);
    }
    st_site(site_ptr(din, warp, vol, y), v);
}

// grad[e] += sum over slices of part[slice][e]  (e over 9*NO entries), in FP64: eight threads per entry,
// each over every eighth slice, added in a fixed order (one thread per entry walked 128 slices: 40 us)
__global__ void __launch_bounds__(256)
k_g_reduce_w(const float2* __restrict__ part, int nslice, int ne, double2* __restrict__ grad) {
    __shared__ double2 sh[8][32];
    const int el = threadIdx.x & 31, q = threadIdx.x >> 5;
    const int e = blockIdx.x * 32 + el;
    double re = 0.0, im = 0.0;
    if (e < ne)
        for (int p = q; p < nslice; p += 8) {
            const float2 z = part[(size_t)p * ne + e];
            re += z.x;
            im += z.y;
        }
    sh[q][el] = make_double2(re, im);
    __syncthreads();
    if (q == 0 && e < ne) {
        for (int k = 1; k < 8; k++) {
            re += sh[k][el].x;
            im += sh[k][el].y;
        }
        grad[e].x += re;
        grad[e].y += im;
    }
}

// byte offset of (row r, 16-byte chunk j) in a tile of 128-byte rows with 128-byte swizzle
__device__ __forceinline__ uint32_t sw128(int r, int j) {
    return (uint32_t)((r >> 3) * 1024 + (r & 7) * 128 + ((j ^ (r & 7)) << 4));
}

// ---------------------------------------------------------------------------
// backward to the weights on tcgen05:
//   dW[d][co][ci][s][s'] = sum_{x,c} dout[co](x)[s][c] conj(g_d(a_ci)(x)[s'][c])
// as real GEMMs with K = (site, colour): P[n][m] = sum g[n] dout[m], n = (ci, s', re/im), m = (co, s, re/im);
// Re = P[r][r] + P[i][i], Im = P[r][i] - P[i][r].  Both operands are MN-major: a tile row is one site's 64 real
// entries of one colour, which is how a thread (site, channel) has them, one 16-byte chunk.
// dout is bf16.  The transported activations g are FP32 and stay so: they enter as three bf16 terms
// hi + mid + lo (24 bits) in two MMAs, [hi; mid] in the 128 rows of A and [lo; 0] on top.  The FP32 sums of TMEM
// run over TW_FLUSH tiles (24 accumulations each) and are then added to this CTA's partial in FP32, so that
// a chain is no longer than the 3072-term FP32 chains of the SIMT kernel this replaced; k_g_reduce_w adds the
// partials in FP64.
// One CTA: 32-site tiles of a slice, 256 threads = 32 sites x 8 channels, directions 3y .. 3y+2 (CI = 8) or, for one
// input channel (CI = 1), directions 1..8 in the place of the channels and direction 0 after them.  Two stage
// buffers (36 KB each): the transport of the next direction overlaps the MMAs of this one, and the loads of the
// one after are in flight; two CTAs per SM fill each other's barrier waits.  The transport and the splitting
// bound it (640 instructions per 32 sites, channel and direction).
// 16^3 x 32: 8 -> 8 layer 2137 us on SIMT (the gather and 32 x 32 complex products per site from shared memory),
// 8 -> 1 776 us, 1 -> 8 688 us; here 332, 290 and 68 us.
// ---------------------------------------------------------------------------
constexpr int TW_SITES = 32;
constexpr int TW_THREADS = TW_SITES * 8;
constexpr int TW_FLUSH = 8;
constexpr uint32_t TW_TILE = TW_SITES * 128;             // 32 rows x 64 bf16
constexpr uint32_t TW_STAGE = 9 * TW_TILE;               // 3 colours x (hi, mid, lo)
constexpr uint32_t TW_SMEM = 2 * TW_STAGE + 2 * 3 * TW_TILE + TW_TILE + 1024 + 64;

template <int CI, int CO>
__global__ void __launch_bounds__(TW_THREADS, 2)
k_g_tw(Geom gm, const float2* __restrict__ u, const bf2* __restrict__ a, const bf2* __restrict__ dout,
       float* __restrict__ part, int* __restrict__ err) {
    using namespace tc;
    extern __shared__ uint8_t smem_raw[];
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
    uint8_t* sG = smem;                                    // [2][3 colours][hi, mid, lo]
    uint8_t* sD = sG + 2 * TW_STAGE;                       // [2][3 colours]
    uint8_t* sZ = sD + 2 * 3 * TW_TILE;                    // zeros
    uint64_t* done = reinterpret_cast<uint64_t*>(sZ + TW_TILE);   // [2]
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(done + 2);
    volatile int* s_fail = reinterpret_cast<volatile int*>(tmem_slot + 1);
    constexpr int ND = CI == 8 ? 3 : 2;                    // stages per tile
    constexpr int NO = CO * CI * 16;
    constexpr int NCOL = CO == 8 ? 64 : 16;                // columns of the MMA (8 used when CO = 1)
    const int vol = gm.vol;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        mbar_init(&done[0], 1);
        mbar_init(&done[1], 1);
        *s_fail = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     ::"r"(smem_u32(tmem_slot)), "r"(256u));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    for (int i = threadIdx.x; i < (int)(TW_TILE / 16); i += blockDim.x)
        reinterpret_cast<uint4*>(sZ)[i] = make_uint4(0, 0, 0, 0);
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem_d = *tmem_slot;

    const int row = threadIdx.x & (TW_SITES - 1), ch = threadIdx.x / TW_SITES;
    const int ntiles = (vol + TW_SITES - 1) / TW_SITES;
    auto dir = [&](int dl) { return CI == 8 ? (int)blockIdx.y * 3 + dl : dl == 0 ? 1 + ch : 0; };
    // the loads of a stage are issued one stage ahead (dead sites load site 0)
    auto fetch = [&](HopLoad<1>& p, int t, int dl) {
        const int x = t * TW_SITES + row;
        if (t < ntiles && (CI == 8 || dl == 0 || ch == 0))
            hop_load<false, 1>(p, gm, u, a, CI == 8 ? ch : 0, x < vol ? x : 0, dir(dl));
    };
    int q = 0, tcount = 0;
    bool first = true, ok = true;
    HopLoad<1> pre;
    fetch(pre, blockIdx.x, 0);
    for (int t = blockIdx.x; t < ntiles && ok; t += gridDim.x, tcount++) {
        const int x = t * TW_SITES + row;
        const bool live = x < vol;
        const uint32_t dbase = (tcount & 1) * 3 * TW_TILE;
        for (int dl = 0; dl < ND; dl++, q++) {
            const int b = q & 1;
            // the MMAs that read buffer b (stage q - 2) and everything before them are done
            if (q >= 2 && !mbar_wait(&done[b], (uint32_t)((q - 2) >> 1) & 1u)) *s_fail = 1;
            __syncthreads();
            if (*s_fail) {
                ok = false;
                break;
            }
            if (dl == 0 && ch < CO) {
                float2 v[12];
                uint4 w[3] = {};
                if (live) {
                    ld_site(site_ptr(dout, ch, vol, x), v);   // bf16 values: packing them again is exact
#pragma unroll
                    for (int c = 0; c < 3; c++)
                        w[c] = make_uint4(pack_bf2(v[c]), pack_bf2(v[3 + c]), pack_bf2(v[6 + c]), pack_bf2(v[9 + c]));
                }
#pragma unroll
                for (int c = 0; c < 3; c++)
                    *reinterpret_cast<uint4*>(sD + dbase + c * TW_TILE + sw128(row, ch)) = w[c];
            }
            if (CI == 8 || dl == 0 || ch == 0) {
                float2 v[12], g[12];
                unpack_site(pre.act[0], v);
                if (dir(dl) == 0) {
#pragma unroll
                    for (int k = 0; k < 12; k++) g[k] = v[k];
                } else {
                    float2 m[9];
                    hop_matrix(pre, m);
#pragma unroll
                    for (int s = 0; s < 4; s++) colour_mul(m, &v[3 * s], &g[3 * s]);
                }
                if (!live) {
#pragma unroll
                    for (int k = 0; k < 12; k++) g[k] = make_float2(0.f, 0.f);
                }
                if (dl + 1 < ND) fetch(pre, t, dl + 1);
                else fetch(pre, t + gridDim.x, 0);
                uint8_t* sb = sG + b * TW_STAGE;
#pragma unroll
                for (int c = 0; c < 3; c++) {
                    unsigned w[3][4];
#pragma unroll
                    for (int s = 0; s < 4; s++) {
                        float2 r = g[3 * s + c];
#pragma unroll
                        for (int k = 0; k < 3; k++) {
                            w[k][s] = pack_bf2(r);
                            const float2 h = unpack_bf2(w[k][s]);
                            r = make_float2(r.x - h.x, r.y - h.y);
                        }
                    }
#pragma unroll
                    for (int k = 0; k < 3; k++)
                        *reinterpret_cast<uint4*>(sb + (3 * c + k) * TW_TILE + sw128(row, ch)) =
                            make_uint4(w[k][0], w[k][1], w[k][2], w[k][3]);
                }
            } else {
                fetch(pre, t + gridDim.x, 0);
            }
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            __syncthreads();
            if (threadIdx.x == 0) {
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                constexpr uint32_t idesc = umma_idesc_bf16(NCOL, 128) | UMMA_MN_MAJOR_AB;
#pragma unroll
                for (int c = 0; c < 3; c++) {
                    const uint32_t hi = smem_u32(sG + b * TW_STAGE + 3 * c * TW_TILE), lo = hi + 2 * TW_TILE;
                    const uint32_t dd = smem_u32(sD + dbase + c * TW_TILE);
#pragma unroll
                    for (int kk = 0; kk < TW_SITES / 16; kk++) {
                        const uint64_t db = umma_desc_mn_sw128(dd + kk * 2048, TW_TILE);
                        umma_bf16(tmem_d + (uint32_t)(dl * 64), umma_desc_mn_sw128(hi + kk * 2048, TW_TILE), db, idesc,
                                  (first && c == 0 && kk == 0) ? 0u : 1u);
                        umma_bf16(tmem_d + (uint32_t)(dl * 64),
                                  umma_desc_mn_sw128(lo + kk * 2048, smem_u32(sZ) - lo - kk * 2048), db, idesc, 1u);
                    }
                }
                umma_commit(&done[b]);
            }
        }
        if (!ok) break;
        first = false;
        const bool last = t + (int)gridDim.x >= ntiles;
        if (tcount % TW_FLUSH == TW_FLUSH - 1 || last) {
            if (!mbar_wait(&done[(q - 1) & 1], (uint32_t)((q - 1) >> 1) & 1u)) *s_fail = 1;
            __syncwarp();
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const int lg = warp & 3;   // TMEM lanes of this warp; warps w and w + 4 share the columns
            const int r = lg * 32 + lane, n = r & 63, half = r >> 6;
            const int pt = n & 1, sp = (n >> 1) & 3, cn = n >> 3;
            for (int cq = warp >> 2; cq < (CO == 8 ? 4 : 1); cq += 2) {
                for (int dl = 0; dl < ND; dl++) {
                    float v[16];
                    tmem_ld16<16>(tmem_d + ((uint32_t)(lg * 32) << 16) + (uint32_t)(dl * 64 + cq * 16), v);
                    const int d = CI == 8 ? blockIdx.y * 3 + dl : dl == 0 ? 1 + cn : 0;
                    const int ci = CI == 8 ? cn : 0;
                    const bool used = CI == 8 || dl == 0 || cn == 0;
                    float* out = part + (((size_t)(blockIdx.x * 2 + half) * 9 + d) * NO) * 2 + pt;
#pragma unroll
                    for (int j = 0; j < 8; j++) {
                        // even column: re of dout, odd: im; this lane holds g's re (pt = 0) or im (pt = 1)
                        const float o = __shfl_xor_sync(0xffffffffu, v[2 * j + 1], 1);
                        const float z = pt == 0 ? v[2 * j] + o : o - v[2 * j];
                        const int m = cq * 8 + j, co = m >> 2, s = m & 3;
                        if (used && co < CO) {
                            float* p = out + (size_t)(((co * CI + ci) * 4 + s) * 4 + sp) * 2;
                            *p = tcount < TW_FLUSH ? z : *p + z;
                        }
                    }
                }
            }
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            __syncthreads();
            first = true;
            if (*s_fail) ok = false;
        }
    }
    if (!ok && threadIdx.x == 0) atomicExch(err, SEEDCG_ERR_TIMEOUT);
    // on a timeout MMAs may still be in flight: wait for the last committed group (bounded) before TMEM is freed
    if (!ok && q > 0) mbar_wait(&done[(q - 1) & 1], (uint32_t)((q - 1) >> 1) & 1u);
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_d), "r"(256u));
    }
}

// ---------------------------------------------------------------------------
// layer 2 on tcgen05 (see the file header).  One CTA = 128 sites, 256 threads (four channels each, in two
// pairs; the loads of the next pair are in flight); two CTAs per SM fill each other's barrier waits.
// 16^3 x 32: 313 us with one CTA per SM and every load waited for, 137 us here (bound by the transport's issue).
// MODE 0 (forward):  A = U(x,d) h1_ci(x+d), B = W in real form; epilogue z2, h2 = ReLU(z2).
// MODE 1 (backward through the data): A = adjoint transport of d2_co, B = W^dag in
//        real form; epilogue d1 = D masked by z1 > 0 (real and imaginary parts).
// K of direction d: k = (ch * 4 + spin) * 2 + {re, im} over the 8 channels of the
// input side; N: n = (ch' * 4 + spin') * 2 + {re, im} over the output side.
// ---------------------------------------------------------------------------
constexpr int TC_SITES = 128;
constexpr uint32_t TC_A_BYTES = TC_SITES * 128;      // 128 rows x 64 bf16
constexpr uint32_t TC_B_BYTES = 64 * 128;            // 64 rows x 64 bf16
// no slack for alignment: two CTAs fill the SM's 228 KB (the base is 1024-byte aligned, checked)
constexpr uint32_t TC_SMEM = 2 * 3 * TC_A_BYTES + 2 * TC_B_BYTES + 64;
constexpr uint32_t TC_TMEM_COLS = 256;               // 3 colours x 64 columns

template <int MODE>
__global__ void __launch_bounds__(256, 2)
k_g_tc(Geom gm, const float2* __restrict__ u, const bf2* __restrict__ in, const uint4* __restrict__ wimg,
       const bf2* __restrict__ zprev, bf2* __restrict__ out0, bf2* __restrict__ out1, int* __restrict__ err) {
    using namespace tc;
    extern __shared__ __align__(1024) uint8_t tc_smem[];
    if (smem_u32(tc_smem) & 1023u) {   // the swizzled tiles need it
        if (threadIdx.x == 0) atomicExch(err, SEEDCG_ERR_CUDA);
        return;
    }
    uint8_t* sA = tc_smem;                                   // [2 buffers][3 colours][TC_A_BYTES]
    uint8_t* sB = sA + 2 * 3 * TC_A_BYTES;              // [2 buffers][TC_B_BYTES]
    uint64_t* done = reinterpret_cast<uint64_t*>(sB + 2 * TC_B_BYTES);   // [2]
    uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(done + 2);
    volatile int* s_fail = reinterpret_cast<volatile int*>(tmem_slot + 1);
    const int vol = gm.vol;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int x0 = blockIdx.x * TC_SITES;
    if (threadIdx.x == 0) {
        mbar_init(&done[0], 1);
        mbar_init(&done[1], 1);
        *s_fail = 0;
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     ::"r"(smem_u32(tmem_slot)), "r"(TC_TMEM_COLS));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem_d = *tmem_slot;

    // this thread's site and half of the input channels
    const int row = threadIdx.x & (TC_SITES - 1);
    const int ch0 = 4 * (threadIdx.x >> 7);
    const int x = x0 + row;
    const bool live = x < vol;
    // the loads of a pair of channels (and a direction's link and piece of the weight image) are issued one
    // pair ahead
    static_assert(TC_B_BYTES == 2 * 256 * 16, "two 16-byte pieces of the weight image per thread");
    HopLoad<2> pre;
    hop_load<MODE != 0, 2>(pre, gm, u, in, ch0, live ? x : 0, 0);
    int issued = 0;   // MMA groups committed (one per direction)
    for (int d = 0; d < 9; d++) {
        const int b = d & 1;
        if (d >= 2) {
            // the MMAs that read buffer b (direction d - 2) must be done before it is refilled
            if (!mbar_wait(&done[b], (uint32_t)((d - 2) >> 1) & 1u)) *s_fail = 1;
        }
        __syncthreads();
        if (*s_fail) break;
        // B: this direction's weights (a ready 128-byte-swizzled image)
        uint4 w0, w1;
        {
            const uint4* src = wimg + (size_t)d * (TC_B_BYTES / 16) + threadIdx.x;
            w0 = __ldg(src);
            w1 = __ldg(src + 256);
        }
        // A: the transported activations of channels ch0 .. ch0 + 3 at this site
        float2 m[9];
        if (d > 0) hop_matrix(pre, m);
        const int src_site = hop_from<MODE != 0>(gm, live ? x : 0, d).src;
#pragma unroll
        for (int pr = 0; pr < 2; pr++) {
            float2 v[2][12];
            unpack_site(pre.act[0], v[0]);
            unpack_site(pre.act[1], v[1]);
            if (pr == 0) {
#pragma unroll
                for (int k = 0; k < 2; k++) {
                    const uint4* q = reinterpret_cast<const uint4*>(site_ptr(in, ch0 + 2 + k, vol, src_site));
#pragma unroll
                    for (int j = 0; j < 3; j++) pre.act[k][j] = __ldg(q + j);
                }
            } else if (d < 8) {
                hop_load<MODE != 0, 2>(pre, gm, u, in, ch0, live ? x : 0, d + 1);
            }
#pragma unroll
            for (int q = 0; q < 2; q++) {
                float2 g[12];
                if (d == 0) {
#pragma unroll
                    for (int k = 0; k < 12; k++) g[k] = v[q][k];
                } else {
#pragma unroll
                    for (int s = 0; s < 4; s++) colour_mul(m, &v[q][3 * s], &g[3 * s]);
                }
                if (!live) {
#pragma unroll
                    for (int k = 0; k < 12; k++) g[k] = make_float2(0.f, 0.f);
                }
                // colour c of this (site, channel): 4 spins x (re, im) = 16 bytes, chunk ch of the row
#pragma unroll
                for (int c = 0; c < 3; c++) {
                    const uint4 w = make_uint4(pack_bf2(g[c]), pack_bf2(g[3 + c]), pack_bf2(g[6 + c]), pack_bf2(g[9 + c]));
                    *reinterpret_cast<uint4*>(sA + (b * 3 + c) * TC_A_BYTES + sw128(row, ch0 + 2 * pr + q)) = w;
                }
            }
        }
        reinterpret_cast<uint4*>(sB + b * TC_B_BYTES)[threadIdx.x] = w0;
        reinterpret_cast<uint4*>(sB + b * TC_B_BYTES)[threadIdx.x + 256] = w1;
        // the tensor cores read shared memory through the async proxy
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncthreads();
        if (threadIdx.x == 0) {
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            constexpr uint32_t idesc = umma_idesc_bf16(64, 128);
            const uint32_t b0 = smem_u32(sB + b * TC_B_BYTES);
#pragma unroll
            for (int c = 0; c < 3; c++) {
                const uint32_t a0 = smem_u32(sA + (b * 3 + c) * TC_A_BYTES);
#pragma unroll
                for (int kk = 0; kk < 4; kk++)
                    umma_bf16(tmem_d + (uint32_t)(c * 64), umma_desc_sw128(a0 + kk * 32), umma_desc_sw128(b0 + kk * 32),
                              idesc, (d > 0 || kk > 0) ? 1u : 0u);
            }
            umma_commit(&done[b]);
        }
        issued = d + 1;
    }
    // the last group's completion covers every earlier MMA of this CTA
    if (issued > 0) {
        const int dl = issued - 1;
        if (!mbar_wait(&done[dl & 1], (uint32_t)(dl >> 1) & 1u)) *s_fail = 1;
    }
    __syncwarp();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    __syncthreads();
    if (*s_fail || issued < 9) {
        if (threadIdx.x == 0) atomicExch(err, SEEDCG_ERR_TIMEOUT);
    } else {
        // warp w reads TMEM lanes [32 (w % 4), + 32), the rows (sites) of its threads, for four output channels
        const int lg = warp & 3, r = lg * 32 + lane;
        const int xs = x0 + r;
        for (int o = 4 * (warp >> 2); o < 4 * (warp >> 2) + 4; o++) {
            float cv[3][8];
#pragma unroll
            for (int c = 0; c < 3; c++)
                tmem_ld8(tmem_d + ((uint32_t)(lg * 32) << 16) + (uint32_t)(c * 64 + o * 8), cv[c]);
            if (xs < vol) {
                float2 z[12];
#pragma unroll
                for (int s = 0; s < 4; s++)
#pragma unroll
                    for (int c = 0; c < 3; c++) z[3 * s + c] = make_float2(cv[c][2 * s], cv[c][2 * s + 1]);
                if (MODE == 0) {
                    float2 hr[12];
#pragma unroll
                    for (int k = 0; k < 12; k++) hr[k] = make_float2(fmaxf(z[k].x, 0.f), fmaxf(z[k].y, 0.f));
                    if (out0) st_site(site_ptr(out0, o, vol, xs), z);   // not kept for inference
                    st_site(site_ptr(out1, o, vol, xs), hr);
                } else {
                    float2 zz[12];
                    ld_site(site_ptr(zprev, o, vol, xs), zz);
#pragma unroll
                    for (int k = 0; k < 12; k++)
                        z[k] = make_float2(zz[k].x > 0.f ? z[k].x : 0.f, zz[k].y > 0.f ? z[k].y : 0.f);
                    st_site(site_ptr(out0, o, vol, xs), z);
                }
            }
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == 0) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_d), "r"(TC_TMEM_COLS));
    }
}

// The B operands of layer 2 as 128-byte-swizzled bf16 images, one 64 x 64 tile per
// direction: forward B[n = (co,s,p)][k = (ci,s',q)] and adjoint B[n = (ci,s',p)][k = (co,s,q)]
// (p, q: 0 real, 1 imaginary), from the FP32 master weights W2[9][8][8][4][4].
__global__ void k_g_wform(const float2* __restrict__ W2, uint8_t* __restrict__ fwd, uint8_t* __restrict__ adj) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;   // one thread per (d, n, k)
    if (t >= 9 * 64 * 64) return;
    const int k = t % 64, n = (t / 64) % 64, d = t / 4096;
    const int q = k & 1, kk = k >> 1, p = n & 1, nn = n >> 1;
    // forward: n -> (co, s), k -> (ci, s')
    {
        const int co = nn >> 2, s = nn & 3, ci = kk >> 2, sp = kk & 3;
        const float2 w = W2[(((size_t)d * 8 + co) * 8 + ci) * 16 + s * 4 + sp];
        const float v = p == 0 ? (q == 0 ? w.x : -w.y) : (q == 0 ? w.y : w.x);
        *reinterpret_cast<unsigned short*>(fwd + (size_t)d * TC_B_BYTES + sw128(n, k >> 3) + (k & 7) * 2) =
            __bfloat16_as_ushort(__float2bfloat16_rn(v));
    }
    // adjoint: n -> (ci, s'), k -> (co, s); din = sum conj(W) dout'
    {
        const int ci = nn >> 2, sp = nn & 3, co = kk >> 2, s = kk & 3;
        const float2 w = W2[(((size_t)d * 8 + co) * 8 + ci) * 16 + s * 4 + sp];
        const float v = p == 0 ? (q == 0 ? w.x : w.y) : (q == 0 ? -w.y : w.x);
        *reinterpret_cast<unsigned short*>(adj + (size_t)d * TC_B_BYTES + sw128(n, k >> 3) + (k & 7) * 2) =
            __bfloat16_as_ushort(__float2bfloat16_rn(v));
    }
}

// ---------------------------------------------------------------------------
// input, output, loss, Adam
// ---------------------------------------------------------------------------
// internal paired-layout index of entry k of site s
__device__ __forceinline__ size_t pidx(int s, int k, int vol) {
    return ((size_t)(k >> 1) * vol + s) * 2 + (k & 1);
}

// a0 = b / ||b|| in bf16 [V][12]
// One thread of a block divides (an FP64 operation takes the pipe 68 clocks per warp, a division a dozen of
// them), and roundings to and from FP32 move bits, with four entries in flight. 16^3 x 32: k_g_scale_in 22.8 -> 16.4 us,
// k_g_loss 47 -> 41 us.
__global__ void k_g_scale_in(const double2* __restrict__ b, const double* __restrict__ nb, bf2* __restrict__ a0,
                             int vol) {
    __shared__ double s_inv;
    if (threadIdx.x == 0) s_inv = 1.0 / *nb;
    __syncthreads();
    const double inv = s_inv;
#pragma unroll 4
    for (long o = blockIdx.x * (long)blockDim.x + threadIdx.x; o < 12L * vol; o += (long)gridDim.x * blockDim.x) {
        const int s = (int)(o / 12), k = (int)(o % 12);
        const double2 z = b[pidx(s, k, vol)];
        a0[o] = __float22bfloat162_rn(make_float2(narrow(z.x * inv), narrow(z.y * inv)));
    }
}

// x0 = ||b|| z3 (FP64 internal layout)
__global__ void k_g_scale_out(const bf2* __restrict__ z3, const double* __restrict__ nb, double2* __restrict__ x0,
                              int vol) {
    const double s = *nb;
#pragma unroll 4
    for (long o = blockIdx.x * (long)blockDim.x + threadIdx.x; o < 12L * vol; o += (long)gridDim.x * blockDim.x) {
        const int st = (int)(o / 12), k = (int)(o % 12);
        const float2 z = __bfloat1622float2(z3[o]);
        x0[pidx(st, k, vol)] = make_double2(s * widen(z.x), s * widen(z.y));
    }
}

// loss term ||y - x||^2 / ||x||^2 / nbatch with y = ||b|| z3, and dz3 = ||b|| * 2 (y - x) / ||x||^2 / nbatch
__global__ void __launch_bounds__(kRedThreads)
k_g_loss(const bf2* __restrict__ z3, const double2* __restrict__ x, const double* __restrict__ nb,
         const double* __restrict__ nx, double inv_batch, bf2* __restrict__ dz3, int vol,
         double* partials, unsigned* ctr, double* loss_acc) {
    const double s = *nb, xn2 = (*nx) * (*nx);
    __shared__ double s_f;
    if (threadIdx.x == 0) s_f = s * 2.0 * inv_batch / xn2;
    __syncthreads();
    const double f = s_f;
    double part = 0.0;
#pragma unroll 4
    for (long o = blockIdx.x * (long)blockDim.x + threadIdx.x; o < 12L * vol; o += (long)gridDim.x * blockDim.x) {
        const int st = (int)(o / 12), k = (int)(o % 12);
        const float2 z = __bfloat1622float2(z3[o]);
        const double2 xv = x[pidx(st, k, vol)];
        const double rx = s * widen(z.x) - xv.x, ry = s * widen(z.y) - xv.y;
        part += rx * rx + ry * ry;
        dz3[o] = __float22bfloat162_rn(make_float2(narrow(f * rx), narrow(f * ry)));
    }
    double red[1] = {part};
    grid_sum<1>(red, partials, ctr, [&](double* tot) { *loss_acc += tot[0] / xn2 * inv_batch; });
}

// Adam on real and imaginary parts: FP32 master weights and moments, FP64 gradient;
// the bf16 copy the layers read is refreshed in the same pass
__global__ void k_g_adam(float2* __restrict__ W, bf2* __restrict__ Wb, const double2* __restrict__ g,
                         float2* __restrict__ m, float2* __restrict__ v, int ne, float lr, float b1, float b2,
                         float eps, float c1, float c2) {
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e >= ne) return;
    const float gx = (float)g[e].x, gy = (float)g[e].y;
    float2 mm = m[e], vv = v[e], w = W[e];
    mm.x = b1 * mm.x + (1.f - b1) * gx;
    mm.y = b1 * mm.y + (1.f - b1) * gy;
    vv.x = b2 * vv.x + (1.f - b2) * gx * gx;
    vv.y = b2 * vv.y + (1.f - b2) * gy * gy;
    w.x -= lr * (mm.x / c1) / (sqrtf(vv.x / c2) + eps);
    w.y -= lr * (mm.y / c1) / (sqrtf(vv.y / c2) + eps);
    m[e] = mm;
    v[e] = vv;
    W[e] = w;
    Wb[e] = __float22bfloat162_rn(w);
}

__global__ void k_g_round(const float2* __restrict__ W, bf2* __restrict__ Wb, int ne) {
    const int e = blockIdx.x * blockDim.x + threadIdx.x;
    if (e < ne) Wb[e] = __float22bfloat162_rn(W[e]);
}

}  // namespace

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------
struct GuessState {
    static constexpr int NW1 = 9 * 8 * 1 * 16, NW2 = 9 * 8 * 8 * 16, NW3 = 9 * 1 * 8 * 16;
    static constexpr int NW = NW1 + NW2 + NW3;
    DevBuf w;       // float2 [NW] master weights
    DevBuf wb;      // bf16x2 [NW] the weights the layers read
    DevBuf wimg;    // layer-2 B operands: forward and adjoint images, 9 x 8 KB each
    DevBuf adam;    // m, v float2 [NW] each
    DevBuf grad;    // double2 [NW]
    DevBuf act;     // activations and gradients (bf16)
    DevBuf part;    // weight-gradient partials
    DevBuf scal;    // norms, loss, the tensor-core error flag
    int steps = 0;
    bool have_weights = false;
};

GuessState* guess_state(seedcg_handle* h) {
    if (!h->guess) h->guess = new GuessState();
    return reinterpret_cast<GuessState*>(h->guess);
}

bool guess_ready(const seedcg_handle* h) {
    return h->guess && reinterpret_cast<const GuessState*>(h->guess)->have_weights;
}

void guess_free(seedcg_handle* h) {
    if (h->guess) {
        GuessState* g = reinterpret_cast<GuessState*>(h->guess);
        delete g;   // every DevBuf frees its allocation
        h->guess = nullptr;
    }
}

namespace {

struct Acts {
    bf2 *a0, *z1, *h1, *z2, *h2, *z3, *d3, *d2, *d1;
    double* nb;
    double* nx;
    double* loss;
    int* tc_err;
};

Acts carve_acts(GuessState* G, int vol) {
    const size_t site = (size_t)vol * 12;   // bf16x2 entries of one channel
    const size_t need = site * (1 + 8 * 4 + 1 + 1 + 8 * 2) * sizeof(bf2) + 4096;
    G->act.ensure(need);
    G->scal.ensure(64 * sizeof(double) + 8192 * sizeof(double) + 8192 * sizeof(unsigned));
    bf2* p = G->act.as<bf2>();
    Acts A;
    A.a0 = p; p += site;
    A.z1 = p; p += 8 * site;
    A.h1 = p; p += 8 * site;
    A.z2 = p; p += 8 * site;
    A.h2 = p; p += 8 * site;
    A.z3 = p; p += site;
    A.d3 = p; p += site;
    A.d2 = p; p += 8 * site;
    A.d1 = p; p += 8 * site;
    A.nb = G->scal.as<double>();
    A.nx = A.nb + 1;
    A.loss = A.nb + 2;
    A.tc_err = reinterpret_cast<int*>(A.nb + 3);
    return A;
}

// layer 2 on the tensor cores (mode 0 forward, 1 backward through the data)
void layer2_tc(seedcg_handle* h, GuessState* G, int mode, const bf2* in, const bf2* zprev, bf2* out0, bf2* out1,
               int* err, cudaStream_t st) {
    const Geom& gm = h->g;
    const int blocks = (gm.vol + TC_SITES - 1) / TC_SITES;
    const uint4* img = reinterpret_cast<const uint4*>(G->wimg.as<uint8_t>() + (mode ? 9 * TC_B_BYTES : 0));
    if (mode == 0) allow_smem<k_g_tc<0>>(TC_SMEM);
    else allow_smem<k_g_tc<1>>(TC_SMEM);
    if (mode == 0)
        k_g_tc<0><<<blocks, 256, TC_SMEM, st>>>(gm, h->u32.as<float2>(), in, img, zprev, out0, out1, err);
    else
        k_g_tc<1><<<blocks, 256, TC_SMEM, st>>>(gm, h->u32.as<float2>(), in, img, zprev, out0, out1, err);
    SEEDCG_CHECK_LAUNCH();
}

// the bf16 weights and the layer-2 operand images from the master weights
void refresh_weight_forms(GuessState* G, cudaStream_t st) {
    uint8_t* img = G->wimg.as<uint8_t>();
    k_g_wform<<<(9 * 64 * 64 + 255) / 256, 256, 0, st>>>(G->w.as<float2>() + GuessState::NW1, img, img + 9 * TC_B_BYTES);
    SEEDCG_CHECK_LAUNCH();
}

void check_tc(const Acts& A, cudaStream_t st) {
    int e = 0;
    SEEDCG_CUDA_TRY(cudaMemcpyAsync(&e, A.tc_err, sizeof(int), cudaMemcpyDeviceToHost, st));
    SEEDCG_CUDA_TRY(cudaStreamSynchronize(st));
    if (e) throw Error{SEEDCG_ERR_TIMEOUT, "a tensor-core wait of the learned guess expired"};
}

// keep_z: the backward pass will need the pre-activations z1, z2
void forward(seedcg_handle* h, GuessState* G, const Acts& A, const double2* b64, bool keep_z, cudaStream_t st) {
    const Geom& gm = h->g;
    const long n = 12L * gm.vol;
    const float2* u = h->u32.as<float2>();
    const bf2* W = G->wb.as<bf2>();
    double* partials = A.nb + 64;
    unsigned* ctr = reinterpret_cast<unsigned*>(partials + 8192);
    k_norm2_public(b64, n, partials, ctr, A.nb, st);
    k_g_scale_in<<<std::min<long>((n + 255) / 256, 8 * 152), 256, 0, st>>>(b64, A.nb, A.a0, gm.vol);
    SEEDCG_CHECK_LAUNCH();
    const int tiles = (gm.vol + SL - 1) / SL;
    k_g_first<<<tiles, 288, 0, st>>>(gm, u, W, A.a0, keep_z ? A.z1 : nullptr, A.h1);
    SEEDCG_CHECK_LAUNCH();
    layer2_tc(h, G, 0, A.h1, nullptr, keep_z ? A.z2 : nullptr, A.h2, A.tc_err, st);
    allow_smem<k_g_last>(kLastSmem);
    k_g_last<<<tiles, kLastThreads, kLastSmem, st>>>(gm, u, W + GuessState::NW1 + GuessState::NW2, A.h2, A.z3);
    SEEDCG_CHECK_LAUNCH();
}

template <int CI, int CO>
void weight_grad(seedcg_handle* h, GuessState* G, const bf2* a, const bf2* dout, double2* grad, int* err,
                 cudaStream_t st) {
    const Geom& gm = h->g;
    // two CTAs per SM: the directions' three groups share the chip (CI = 8)
    const int ntiles = (gm.vol + TW_SITES - 1) / TW_SITES;
    const int groups = CI == 8 ? 3 : 1;
    const int nslice = std::min(ntiles, 304 / groups);
    constexpr int NO = CO * CI * 16;
    const size_t ne = (size_t)9 * NO;
    G->part.ensure((size_t)nslice * 2 * ne * sizeof(float2));
    allow_smem<k_g_tw<CI, CO>>(TW_SMEM);
    k_g_tw<CI, CO><<<dim3(nslice, groups), TW_THREADS, TW_SMEM, st>>>(gm, h->u32.as<float2>(), a, dout, G->part.as<float>(), err);
    SEEDCG_CHECK_LAUNCH();
    k_g_reduce_w<<<(int)((ne + 31) / 32), 256, 0, st>>>(G->part.as<float2>(), 2 * nslice, (int)ne, grad);
    SEEDCG_CHECK_LAUNCH();
}

// accumulate the loss and gradient of one pair into G->grad / A.loss
void backward_pair(seedcg_handle* h, GuessState* G, const Acts& A, const double2* x64, double inv_batch,
                   cudaStream_t st) {
    const Geom& gm = h->g;
    const long n = 12L * gm.vol;
    const float2* u = h->u32.as<float2>();
    const bf2* W = G->wb.as<bf2>();
    double2* grad = G->grad.as<double2>();
    double* partials = A.nb + 64;
    unsigned* ctr = reinterpret_cast<unsigned*>(partials + 8192);
    k_norm2_public(x64, n, partials, ctr, A.nx, st);
    k_g_loss<<<std::min<long>((n + 1023) / 1024, 4 * 152), kRedThreads, 0, st>>>(A.z3, x64, A.nb, A.nx, inv_batch,
                                                                             A.d3, gm.vol, partials, ctr + 1, A.loss);
    SEEDCG_CHECK_LAUNCH();
    // layer 3 (8 -> 1)
    weight_grad<8, 1>(h, G, A.h2, A.d3, grad + GuessState::NW1 + GuessState::NW2, A.tc_err, st);
    k_g_bwd_data<<<(gm.vol + SL - 1) / SL, 256, 0, st>>>(gm, u, W + GuessState::NW1 + GuessState::NW2, A.d3, A.z2,
                                                         A.d2);
    SEEDCG_CHECK_LAUNCH();
    // layer 2 (8 -> 8)
    weight_grad<8, 8>(h, G, A.h1, A.d2, grad + GuessState::NW1, A.tc_err, st);
    layer2_tc(h, G, 1, A.d2, A.z1, A.d1, nullptr, A.tc_err, st);
    // layer 1 (1 -> 8): only the weight gradient is needed
    weight_grad<1, 8>(h, G, A.a0, A.d1, grad, A.tc_err, st);
}

}  // namespace

void guess_set_weights(seedcg_handle* h, const double* w, cudaStream_t st) {
    GuessState* G = guess_state(h);
    G->w.ensure(GuessState::NW * sizeof(float2));
    G->wb.ensure(GuessState::NW * sizeof(bf2));
    G->wimg.ensure(2 * 9 * TC_B_BYTES);
    G->adam.ensure(2 * GuessState::NW * sizeof(float2));
    G->grad.ensure(GuessState::NW * sizeof(double2));
    std::vector<float2> hw(GuessState::NW);
    for (int e = 0; e < GuessState::NW; e++) hw[e] = make_float2((float)w[2 * e], (float)w[2 * e + 1]);
    SEEDCG_CUDA_TRY(cudaMemcpyAsync(G->w.p, hw.data(), GuessState::NW * sizeof(float2), cudaMemcpyHostToDevice, st));
    SEEDCG_CUDA_TRY(cudaMemsetAsync(G->adam.p, 0, 2 * GuessState::NW * sizeof(float2), st));
    k_g_round<<<(GuessState::NW + 255) / 256, 256, 0, st>>>(G->w.as<float2>(), G->wb.as<bf2>(), GuessState::NW);
    SEEDCG_CHECK_LAUNCH();
    refresh_weight_forms(G, st);
    SEEDCG_CUDA_TRY(cudaStreamSynchronize(st));
    G->steps = 0;
    G->have_weights = true;
}

void guess_get_weights(seedcg_handle* h, double* w, cudaStream_t st) {
    GuessState* G = guess_state(h);
    if (!G->have_weights) throw Error{SEEDCG_ERR_ARG, "no guess weights set"};
    std::vector<float2> hw(GuessState::NW);
    SEEDCG_CUDA_TRY(cudaMemcpyAsync(hw.data(), G->w.p, GuessState::NW * sizeof(float2), cudaMemcpyDeviceToHost, st));
    SEEDCG_CUDA_TRY(cudaStreamSynchronize(st));
    for (int e = 0; e < GuessState::NW; e++) {
        w[2 * e] = hw[e].x;
        w[2 * e + 1] = hw[e].y;
    }
}

// loss and gradient over npairs (B, X internal FP64 [npairs][n]); grad out in
// complex128 [NW] (host) if non-null; returns the loss
double guess_loss_grad(seedcg_handle* h, int npairs, const double2* B, const double2* X, double* grad_out,
                       cudaStream_t st) {
    GuessState* G = guess_state(h);
    if (!G->have_weights) throw Error{SEEDCG_ERR_ARG, "no guess weights set"};
    const long n = 12L * h->g.vol;
    Acts A = carve_acts(G, h->g.vol);
    SEEDCG_CUDA_TRY(cudaMemsetAsync(G->grad.p, 0, GuessState::NW * sizeof(double2), st));
    SEEDCG_CUDA_TRY(cudaMemsetAsync(A.nb, 0, G->scal.bytes, st));
    for (int k = 0; k < npairs; k++) {
        forward(h, G, A, B + (size_t)k * n, true, st);
        backward_pair(h, G, A, X + (size_t)k * n, 1.0 / npairs, st);
    }
    double loss = 0.0;
    SEEDCG_CUDA_TRY(cudaMemcpyAsync(&loss, A.loss, sizeof(double), cudaMemcpyDeviceToHost, st));
    if (grad_out)
        SEEDCG_CUDA_TRY(cudaMemcpyAsync(grad_out, G->grad.p, GuessState::NW * sizeof(double2), cudaMemcpyDeviceToHost, st));
    check_tc(A, st);
    return loss;
}

// Adam training over `epochs` passes of the pairs in order, mini-batches of `batch`
double guess_train(seedcg_handle* h, int npairs, const double2* B, const double2* X, int epochs, int batch,
                   double lr, cudaStream_t st) {
    GuessState* G = guess_state(h);
    double last = 0.0;
    for (int ep = 0; ep < epochs; ep++) {
        double tot = 0.0;
        for (int k0 = 0; k0 < npairs; k0 += batch) {
            const int nb = std::min(batch, npairs - k0);
            const double l = guess_loss_grad(h, nb, B + (size_t)k0 * 12 * h->g.vol, X + (size_t)k0 * 12 * h->g.vol,
                                             nullptr, st);
            tot += l * nb;
            G->steps++;
            const float b1 = 0.9f, b2 = 0.999f;
            const float c1 = 1.f - powf(b1, (float)G->steps), c2 = 1.f - powf(b2, (float)G->steps);
            float2* m = G->adam.as<float2>();
            k_g_adam<<<(GuessState::NW + 255) / 256, 256, 0, st>>>(G->w.as<float2>(), G->wb.as<bf2>(),
                                                                  G->grad.as<double2>(), m, m + GuessState::NW,
                                                                  GuessState::NW, (float)lr, b1, b2, 1e-8f, c1, c2);
            SEEDCG_CHECK_LAUNCH();
            refresh_weight_forms(G, st);
        }
        last = tot / npairs;
    }
    SEEDCG_CUDA_TRY(cudaStreamSynchronize(st));
    return last;
}

// x0 = net(b) for n fields (internal FP64 in/out)
void guess_predict(seedcg_handle* h, int n_fields, const double2* B, double2* X0, cudaStream_t st) {
    GuessState* G = guess_state(h);
    if (!G->have_weights) throw Error{SEEDCG_ERR_ARG, "no guess weights set"};
    const long n = 12L * h->g.vol;
    Acts A = carve_acts(G, h->g.vol);
    SEEDCG_CUDA_TRY(cudaMemsetAsync(A.nb, 0, G->scal.bytes, st));
    for (int k = 0; k < n_fields; k++) {
        forward(h, G, A, B + (size_t)k * n, false, st);
        k_g_scale_out<<<std::min<long>((n + 255) / 256, 8 * 152), 256, 0, st>>>(A.z3, A.nb, X0 + (size_t)k * n,
                                                                            h->g.vol);
        SEEDCG_CHECK_LAUNCH();
    }
    check_tc(A, st);
}

}  // namespace seedcg
