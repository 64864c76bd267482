// Device-side Wilson hopping term, shared by the dslash kernels and the fused
// solver kernels.
//
//   (D psi)(x) = psi(x) - kappa sum_mu [ P-_mu U_mu(x) psi(x+mu) s_f
//                                      + P+_mu U_mu(x-mu)^dag psi(x-mu) s_b ]
//   P-_mu = 1 - g_mu,  P+_mu = 1 + g_mu,  s = -1 on hops that wrap t.
//   D^dag = g5 D g5 swaps P- and P+ (g5 anticommutes with every g_mu).
//
// Each projector has rank 2 in spin space, so a hop projects the 4-spinor to
// two colour vectors h0, h1, multiplies them by the link and rebuilds the
// other two spin components from them.  In the chiral basis
// g_k = [[0,-i s_k],[i s_k,0]], g_4 = [[0,1],[1,0]] the projections for
// P = 1 + S g_mu (S = +-1) are
//   mu=x: h0 = p0 - S i p3, h1 = p1 - S i p2;  full = (r0, r1,  S i r1,  S i r0)
//   mu=y: h0 = p0 - S   p3, h1 = p1 + S   p2;  full = (r0, r1,  S   r1, -S   r0)
//   mu=z: h0 = p0 - S i p2, h1 = p1 + S i p3;  full = (r0, r1,  S i r0, -S i r1)
//   mu=t: h0 = p0 + S   p2, h1 = p1 + S   p3;  full = (r0, r1,  S   r0,  S   r1)
#pragma once

#include <type_traits>

#include "internal.cuh"

namespace seedcg {

template <typename R> struct Spinor { cx_t<R> c[4][3]; };

// h = (1 + S g_mu) p, two colour vectors
template <int MU, int S, typename R>
__device__ __forceinline__ void spin_project(const Spinor<R>& p, cx_t<R> h[2][3]) {
#pragma unroll
    for (int a = 0; a < 3; a++) {
        if (MU == 0) {
            h[0][a] = S > 0 ? csub(p.c[0][a], ci(p.c[3][a])) : cadd(p.c[0][a], ci(p.c[3][a]));
            h[1][a] = S > 0 ? csub(p.c[1][a], ci(p.c[2][a])) : cadd(p.c[1][a], ci(p.c[2][a]));
        } else if (MU == 1) {
            h[0][a] = S > 0 ? csub(p.c[0][a], p.c[3][a]) : cadd(p.c[0][a], p.c[3][a]);
            h[1][a] = S > 0 ? cadd(p.c[1][a], p.c[2][a]) : csub(p.c[1][a], p.c[2][a]);
        } else if (MU == 2) {
            h[0][a] = S > 0 ? csub(p.c[0][a], ci(p.c[2][a])) : cadd(p.c[0][a], ci(p.c[2][a]));
            h[1][a] = S > 0 ? cadd(p.c[1][a], ci(p.c[3][a])) : csub(p.c[1][a], ci(p.c[3][a]));
        } else {
            h[0][a] = S > 0 ? cadd(p.c[0][a], p.c[2][a]) : csub(p.c[0][a], p.c[2][a]);
            h[1][a] = S > 0 ? cadd(p.c[1][a], p.c[3][a]) : csub(p.c[1][a], p.c[3][a]);
        }
    }
}

// acc += coef * (full spinor rebuilt from r) for P = 1 + S g_mu
template <int MU, int S, typename R, bool SCALE = true>
__device__ __forceinline__ void spin_accum(Spinor<R>& acc, const cx_t<R> r[2][3], R coef) {
#pragma unroll
    for (int a = 0; a < 3; a++) {
        cx_t<R> r0 = SCALE ? cscale(r[0][a], coef) : r[0][a];
        cx_t<R> r1 = SCALE ? cscale(r[1][a], coef) : r[1][a];
        acc.c[0][a] = cadd(acc.c[0][a], r0);
        acc.c[1][a] = cadd(acc.c[1][a], r1);
        if (MU == 0) {
            acc.c[2][a] = S > 0 ? cadd(acc.c[2][a], ci(r1)) : csub(acc.c[2][a], ci(r1));
            acc.c[3][a] = S > 0 ? cadd(acc.c[3][a], ci(r0)) : csub(acc.c[3][a], ci(r0));
        } else if (MU == 1) {
            acc.c[2][a] = S > 0 ? cadd(acc.c[2][a], r1) : csub(acc.c[2][a], r1);
            acc.c[3][a] = S > 0 ? csub(acc.c[3][a], r0) : cadd(acc.c[3][a], r0);
        } else if (MU == 2) {
            acc.c[2][a] = S > 0 ? cadd(acc.c[2][a], ci(r0)) : csub(acc.c[2][a], ci(r0));
            acc.c[3][a] = S > 0 ? csub(acc.c[3][a], ci(r1)) : cadd(acc.c[3][a], ci(r1));
        } else {
            acc.c[2][a] = S > 0 ? cadd(acc.c[2][a], r0) : csub(acc.c[2][a], r0);
            acc.c[3][a] = S > 0 ? cadd(acc.c[3][a], r1) : csub(acc.c[3][a], r1);
        }
    }
}

// ||v||^2 at one site, in the working precision
template <typename R>
__device__ __forceinline__ R spinor_norm2(const Spinor<R>& v) {
    R a = 0;
#pragma unroll
    for (int k = 0; k < 12; k++) {
        const cx_t<R> z = v.c[k / 3][k % 3];
        a += z.x * z.x + z.y * z.y;
    }
    return a;
}

// ---------------------------------------------------------------------------
// spinor loads/stores in the internal layouts
// ---------------------------------------------------------------------------
// flat complex index of spinor element k (0..11) of site s
__host__ __device__ __forceinline__ size_t sidx(int k, int s, int vol) {
    return ((size_t)(k >> 1) * (size_t)vol + (size_t)s) * 2 + (size_t)(k & 1);
}

__device__ __forceinline__ void load_spinor(const float2* p, int vol, int s,
                                            Spinor<float>& out) {
    const float4* q = reinterpret_cast<const float4*>(p) + s;
#pragma unroll
    for (int c = 0; c < 6; c++) {
        const float4 z = q[(size_t)c * vol];
        out.c[(2 * c) / 3][(2 * c) % 3] = make_float2(z.x, z.y);
        out.c[(2 * c + 1) / 3][(2 * c + 1) % 3] = make_float2(z.z, z.w);
    }
}
__device__ __forceinline__ void store_spinor(float2* __restrict__ p, int vol, int s,
                                             const Spinor<float>& v) {
    float4* q = reinterpret_cast<float4*>(p) + s;
#pragma unroll
    for (int c = 0; c < 6; c++) {
        const float2 a = v.c[(2 * c) / 3][(2 * c) % 3], b = v.c[(2 * c + 1) / 3][(2 * c + 1) % 3];
        q[(size_t)c * vol] = make_float4(a.x, a.y, b.x, b.y);
    }
}
// The warp's index within its block, computed so that the compiler knows it is the same for all lanes: what
// depends on it (the right-hand side, its field's plane addresses) then lives in uniform registers, and a gather is
// one load at [uniform plane base + 32-bit lane offset] without 64-bit address arithmetic per plane.
__device__ __forceinline__ int uniform_warp(int w) { return __shfl_sync(0xffffffffu, w, 0); }
// neighbour of a site in each direction, as byte offsets (16 * site) of the gathers
struct OffNbr {
    unsigned f[4], b[4];
};
// spinor at byte offset `off` (16 * site) of an FP32 field whose planes are `plane` bytes apart
__device__ __forceinline__ void load_spinor_at(const char* field, size_t plane, unsigned off, Spinor<float>& out) {
#pragma unroll
    for (int c = 0; c < 6; c++) {
        const float4 z = *reinterpret_cast<const float4*>(field + c * plane + off);
        out.c[(2 * c) / 3][(2 * c) % 3] = make_float2(z.x, z.y);
        out.c[(2 * c + 1) / 3][(2 * c + 1) % 3] = make_float2(z.z, z.w);
    }
}
__device__ __forceinline__ void store_spinor_at(char* field, size_t plane, unsigned off, const Spinor<float>& v) {
#pragma unroll
    for (int c = 0; c < 6; c++) {
        const float2 a = v.c[(2 * c) / 3][(2 * c) % 3], b = v.c[(2 * c + 1) / 3][(2 * c + 1) % 3];
        *reinterpret_cast<float4*>(field + c * plane + off) = make_float4(a.x, a.y, b.x, b.y);
    }
}
__device__ __forceinline__ void load_spinor(const double2* p, int vol, int s,
                                            Spinor<double>& out) {
#pragma unroll
    for (int k = 0; k < 12; k++) out.c[k / 3][k % 3] = p[sidx(k, s, vol)];
}
__device__ __forceinline__ void store_spinor(double2* __restrict__ p, int vol, int s,
                                             const Spinor<double>& v) {
#pragma unroll
    for (int k = 0; k < 12; k++) p[sidx(k, s, vol)] = v.c[k / 3][k % 3];
}

// an FP32 spinor widened into the boundary's complex128 layout at site record `rec`
__device__ __forceinline__ void put_spinor_f64(const OutF64& o, size_t rec, const Spinor<float>& v) {
    double* q = o.p + rec * 24;
    if (o.wide) {
#pragma unroll
        for (int c = 0; c < 6; c++) {
            const float2 a = v.c[(2 * c) / 3][(2 * c) % 3], b = v.c[(2 * c + 1) / 3][(2 * c + 1) % 3];
            asm volatile("st.global.v4.f64 [%0], {%1, %2, %3, %4};" ::"l"(q + 4 * c), "d"((double)a.x),
                         "d"((double)a.y), "d"((double)b.x), "d"((double)b.y) : "memory");
        }
    } else {
#pragma unroll
        for (int k = 0; k < 12; k++)
            reinterpret_cast<double2*>(q)[k] = make_double2((double)v.c[k / 3][k % 3].x, (double)v.c[k / 3][k % 3].y);
    }
}

// ---------------------------------------------------------------------------
// neighbours
// ---------------------------------------------------------------------------
struct Nbr {
    int f[4], b[4];
    bool fwrap_t, bwrap_t;
};

__device__ __forceinline__ Nbr neighbours(const Geom& g, int s) {
    Nbr n;
    int c[4];
    int r = s;
    c[0] = r % g.L[0]; r /= g.L[0];
    c[1] = r % g.L[1]; r /= g.L[1];
    c[2] = r % g.L[2]; r /= g.L[2];
    c[3] = r;
#pragma unroll
    for (int mu = 0; mu < 4; mu++) {
        n.f[mu] = (c[mu] == g.L[mu] - 1) ? s - (g.L[mu] - 1) * g.stride[mu] : s + g.stride[mu];
        n.b[mu] = (c[mu] == 0) ? s + (g.L[mu] - 1) * g.stride[mu] : s - g.stride[mu];
    }
    n.fwrap_t = (c[3] == g.L[3] - 1);
    n.bwrap_t = (c[3] == 0);
    return n;
}

__device__ __forceinline__ OffNbr offsets_of(const Nbr& nb, int shift) {
    OffNbr o;
#pragma unroll
    for (int mu = 0; mu < 4; mu++) {
        o.f[mu] = (unsigned)(nb.f[mu] >> shift) * 16u;
        o.b[mu] = (unsigned)(nb.b[mu] >> shift) * 16u;
    }
    return o;
}

// Staging of a tile's links [fwd/bwd][mu][3a+b][NS sites] in shared memory: a warp takes whole rows (direction, mu, entry), a
// lane a site.  src(dir, mu, j, site, scale) gives the link's site and factor, false for sites past the end.
template <int NS, typename Src>
__device__ __forceinline__ void stage_tile_links(float2* sl, const float2* __restrict__ u, int vol, Src src) {
    static_assert(NS == 32, "a lane per site");
    const int nw = blockDim.x >> 5, j = threadIdx.x & 31;
    for (int row = uniform_warp(threadIdx.x >> 5); row < 72; row += nw) {
        const int dir = row / 36, mu = (row / 9) % 4, c = row % 9;
        float2 z = make_float2(0.f, 0.f);
        unsigned site;
        float scale;
        if (src(dir, mu, j, site, scale)) z = cscale(__ldg(u + (size_t)(mu * 9 + c) * vol + site), scale);
        sl[row * NS + j] = z;
    }
}

// First in each round of a tile kernel's loop over fields: the compiler would otherwise read all 72 links before the
// loop and spill them (632 bytes per thread at 80 registers).
__device__ __forceinline__ void links_stay_shared() { asm volatile("" ::: "memory"); }

// Blocks per SM of the tile kernels with `rpb` warps: between 24 and 32 warps at 64 to 80 registers.  D + D^dag
// on 12 fields of 16^3 x 32 in ms: 3 warps x 9 blocks 0.260, 4 x 7 0.262 (x 6 0.278, x 8 0.264, x 9 0.369: spills), 6 x 5
// 0.264, 8 x 4 0.273, 12 x 2 0.289; three uneven fields 0.279, 0.284, 0.269, 0.284, 0.355; five systems of 10x6x14x12
// 0.036, 0.032, 0.025, 0.023, 0.029.  The autotuner chooses among them.
constexpr int tile_blocks(int rpb) { return rpb <= 3 ? 9 : rpb <= 4 ? 7 : rpb <= 6 ? 5 : rpb <= 8 ? 4 : 2; }

// ---------------------------------------------------------------------------
// one hop: acc += coef * P U psi_nbr  (forward: U = U_mu(x); backward: U = U_mu(x-mu)^dag)
// LinkAt(a, b) returns U[a][b] for the link in use.
// ---------------------------------------------------------------------------
template <int MU, int S, bool BACK, typename R, typename LinkAt, bool SCALE = true>
__device__ __forceinline__ void hop(Spinor<R>& acc, const Spinor<R>& nb, LinkAt link, R coef) {
    cx_t<R> h[2][3], r[2][3];
    spin_project<MU, S>(nb, h);
#pragma unroll
    for (int a = 0; a < 3; a++) {
        cx_t<R> r0 = mk<R>(0, 0), r1 = mk<R>(0, 0);
#pragma unroll
        for (int b = 0; b < 3; b++) {
            if (!BACK) {
                cx_t<R> u = link(a, b);
                r0 = cfma(u, h[0][b], r0);
                r1 = cfma(u, h[1][b], r1);
            } else {
                cx_t<R> u = link(b, a);
                r0 = cfma_conj(u, h[0][b], r0);
                r1 = cfma_conj(u, h[1][b], r1);
            }
        }
        r[0][a] = r0;
        r[1][a] = r1;
    }
    spin_accum<MU, S, R, SCALE>(acc, r, coef);
}

// (D psi)(x) or (D^dag psi)(x) at one site, accumulated straight into `out`
// (out = psi(x), then out += -kappa * s * P U psi(y) hop by hop).
// Fwd(mu, e) / Bwd(mu, e) give element e = 3a+b of U_mu(x) / U_mu(x-mu);
// load(y, sp) loads the spinor at site y.
template <int DAG, typename R, typename LoadNbr, typename Fwd, typename Bwd>
__device__ __forceinline__ void wilson_site(const Nbr& n, int s, LoadNbr load, Fwd fl, Bwd bl,
                                            R kappa, Spinor<R>& out) {
    constexpr int SF = DAG ? 1 : -1;   // forward projector 1 - g (D) or 1 + g (D^dag)
    constexpr int SB = -SF;
    const R mk_ = -kappa;
    load(s, out);
    Spinor<R> nb;
    load(n.f[0], nb); hop<0, SF, false>(out, nb, [&](int a, int b) { return fl(0, 3 * a + b); }, mk_);
    load(n.b[0], nb); hop<0, SB, true>(out, nb, [&](int a, int b) { return bl(0, 3 * a + b); }, mk_);
    load(n.f[1], nb); hop<1, SF, false>(out, nb, [&](int a, int b) { return fl(1, 3 * a + b); }, mk_);
    load(n.b[1], nb); hop<1, SB, true>(out, nb, [&](int a, int b) { return bl(1, 3 * a + b); }, mk_);
    load(n.f[2], nb); hop<2, SF, false>(out, nb, [&](int a, int b) { return fl(2, 3 * a + b); }, mk_);
    load(n.b[2], nb); hop<2, SB, true>(out, nb, [&](int a, int b) { return bl(2, 3 * a + b); }, mk_);
    load(n.f[3], nb); hop<3, SF, false>(out, nb, [&](int a, int b) { return fl(3, 3 * a + b); }, n.fwrap_t ? kappa : mk_);
    load(n.b[3], nb); hop<3, SB, true>(out, nb, [&](int a, int b) { return bl(3, 3 * a + b); }, n.bwrap_t ? kappa : mk_);
}

// The eight hops in their order (forward, backward of x, y, z, t) with DEPTH neighbours in flight: step(k, spinor) is
// called for k = 0 .. 7 with the neighbour that load(index) fetched for index(k).
template <int DEPTH, typename R, typename Index, typename LoadNbr, typename Step>
__device__ __forceinline__ void hops_in_flight(Index index, LoadNbr load, Step step) {
    Spinor<R> p[DEPTH];
#pragma unroll
    for (int k = 0; k < DEPTH; k++) load(index(k), p[k]);
#define SEEDCG_STEP(K)                                                                          \
    step(std::integral_constant<int, K>{}, p[K % DEPTH]);                                       \
    if constexpr (K + DEPTH < 8) load(index(K + DEPTH), p[K % DEPTH]);
    SEEDCG_STEP(0)
    SEEDCG_STEP(1)
    SEEDCG_STEP(2)
    SEEDCG_STEP(3)
    SEEDCG_STEP(4)
    SEEDCG_STEP(5)
    SEEDCG_STEP(6)
    SEEDCG_STEP(7)
#undef SEEDCG_STEP
}
template <typename N> __device__ __forceinline__ auto hop_index(const N& n, int k) {
    return (k & 1) ? n.b[k >> 1] : n.f[k >> 1];
}

// wilson_site with DEPTH neighbours in flight, for the FP32 kernels with one thread per site: two where the lattice
// fills the chip (the Lanczos D at 16^3 x 32: 19.3 -> 16.4 us; in FP64 the second spinor's registers cost more than
// they give), four on small lattices, where a thread may have the registers.
// wilson_hops_ahead adds the hops to what `out` holds.
template <int DAG, int DEPTH, typename LoadNbr, typename Fwd, typename Bwd>
__device__ __forceinline__ void wilson_hops_ahead(const Nbr& n, LoadNbr load, Fwd fl, Bwd bl, float kappa,
                                                  Spinor<float>& out) {
    constexpr int SF = DAG ? 1 : -1;
    hops_in_flight<DEPTH, float>(
        [&](int k) { return hop_index(n, k); }, load, [&](auto kk, const Spinor<float>& nb) {
            constexpr int K = decltype(kk)::value, MU = K >> 1, BACK = K & 1;
            if constexpr (BACK)
                hop<MU, -SF, true>(out, nb, [&](int a, int b) { return bl(MU, 3 * a + b); },
                                   MU == 3 && n.bwrap_t ? kappa : -kappa);
            else
                hop<MU, SF, false>(out, nb, [&](int a, int b) { return fl(MU, 3 * a + b); },
                                   MU == 3 && n.fwrap_t ? kappa : -kappa);
        });
}

template <int DAG, int DEPTH, typename LoadNbr, typename Fwd, typename Bwd>
__device__ __forceinline__ void wilson_site_ahead(const Nbr& n, int s, LoadNbr load, Fwd fl, Bwd bl, float kappa,
                                                  Spinor<float>& out) {
    load(s, out);
    wilson_hops_ahead<DAG, DEPTH>(n, load, fl, bl, kappa, out);
}

// Same, with links that already carry the coefficient and the boundary sign (staged that way by the
// tile kernels): out += sum of hops, no scaling.  n.f / n.b are what `load` takes (sites or offsets).
// One neighbour is always in flight while another is multiplied: the gathers' latency bounds these kernels, and
// with the fields' plane addresses in uniform registers the second spinor still leaves 28 warps per SM.
template <int DAG, typename R, typename N, typename LoadNbr, typename Fwd, typename Bwd>
__device__ __forceinline__ void wilson_hops_prescaled(const N& n, LoadNbr load, Fwd fl, Bwd bl, Spinor<R>& out) {
    constexpr int SF = DAG ? 1 : -1;
    hops_in_flight<2, R>([&](int k) { return hop_index(n, k); }, load, [&](auto kk, const Spinor<R>& nb) {
        constexpr int K = decltype(kk)::value, MU = K >> 1, BACK = K & 1;
        auto l = [&](int a, int b) { return BACK ? bl(MU, 3 * a + b) : fl(MU, 3 * a + b); };
        hop<MU, BACK ? -SF : SF, BACK != 0, R, decltype(l), false>(out, nb, l, R(1));
    });
}
// out = psi(s) + sum of hops
template <int DAG, typename R, typename N, typename S, typename LoadNbr, typename Fwd, typename Bwd>
__device__ __forceinline__ void wilson_site_prescaled(const N& n, S s, LoadNbr load, Fwd fl, Bwd bl, Spinor<R>& out) {
    load(s, out);
    wilson_hops_prescaled<DAG, R>(n, load, fl, bl, out);
}

}  // namespace seedcg
