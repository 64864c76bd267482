// The FP64 operator: links in fixed point, D and D^dag on full fields, and the
// even-odd operator of Section 3 on half vectors, all through fix_tile (fixhop.cuh).
#include <algorithm>
#include <cmath>
#include <cstring>

#include "fixhop.cuh"
#include "handle.cuh"

namespace seedcg {
namespace {

// largest and smallest nonzero link component magnitude by link (upper word of the FP64 value:
// 21 bits are enough for a power of two), range[0] a maximum and range[1] a minimum
__global__ void k_fix_range(const double2* __restrict__ u, int vol, unsigned* __restrict__ range) {
    const long t = blockIdx.x * (long)blockDim.x + threadIdx.x;
    unsigned mx = 0;
    if (t < 4L * vol) {
        const int mu = (int)(t / vol), s = (int)(t % vol);
#pragma unroll
        for (int e = 0; e < 9; e++) {
            const double2 z = u[(size_t)(mu * 9 + e) * vol + s];
            mx = max(mx, max((unsigned)__double2hiint(z.x) & 0x7fffffffu, (unsigned)__double2hiint(z.y) & 0x7fffffffu));
        }
    }
    const unsigned hi = __reduce_max_sync(0xffffffffu, mx), lo = __reduce_min_sync(0xffffffffu, mx ? mx : 0x7fffffffu);
    if ((threadIdx.x & 31) == 0) {
        atomicMax(range, hi);
        atomicMin(range + 1, lo);
    }
}

__global__ void k_fix_links(Geom g, const double2* __restrict__ u, double kappa, int k, int4* __restrict__ L) {
    const long t = blockIdx.x * (long)blockDim.x + threadIdx.x;
    if (t >= 36L * g.vol) return;
    const int s = (int)(t % g.vol), mu = (int)(t / g.vol) / 9;
    const double2 z = u[t];
    // hops across the t boundary, forward from the last slice and backward from the first, use this link
    const double c = ldexp(mu == 3 && s / g.stride[3] == g.L[3] - 1 ? kappa : -kappa, k);
    const long long re = __double2ll_rn(c * z.x), im = __double2ll_rn(c * z.y);
    constexpr long long kLow = (1ll << 27) - 1;
    L[t] = make_int4((int)(re >> 27), (int)(re & kLow), (int)(im >> 27), (int)(im & kLow));
}

struct FixStore {
    static constexpr bool kShare = false;
    double2* out;
    FixView v;    // layout of out
    int wide;     // every pair of entries is 32-byte aligned
    __device__ __forceinline__ double operator()(int r, int plane, int idx, int s, bool live, double2 a, double2 b) {
        if (live) {
            double2* q = out + (size_t)r * v.field + (size_t)(v.half ? idx : s) * v.site + (size_t)plane * v.pair;
            if (wide) {
                asm volatile("st.global.v4.f64 [%0], {%1, %2, %3, %4};" ::"l"(q), "d"(a.x), "d"(a.y), "d"(b.x), "d"(b.y)
                             : "memory");
            } else {
                q[0] = a;
                q[1] = b;
            }
        }
        return 0.0;
    }
    __device__ __forceinline__ void put(int, int, double) {}
};

// At most 128 registers: two blocks per SM.  Instruction issue bounds it: 1270 warp instructions per
// 32 sites, direction and field, 216 of them multiply-adds of 32 x 32 + 64 bits and 380 the conversion of the
// neighbour.  16^3 x 32, 12 fields: 898 us between internal fields; 996 us from and to the boundary's spinors, issue 40 %
// busy at 16 warps per SM, DRAM 12 %, where two layout passes took another 303 us.
__global__ void __launch_bounds__(kFixThreads, 2) k_fix_apply(FixDev F, FixOp op, FixStore st, int n) {
    extern __shared__ __align__(16) unsigned char fix_smem[];
    if (!F.ok) {
        fix_plain(F, op, blockIdx.y * gridDim.x + blockIdx.x, gridDim.x * gridDim.y, gridDim.x, n, st);
        return;
    }
    fix_tile(F, op, blockIdx.x, blockIdx.y, n, gridDim.y, fix_smem, st);
}

void fix_go(const FixDev& F, const FixOp& op, double2* out, const FixView& layout, int n, cudaStream_t s) {
    if (n <= 0) return;
    const FixStore st{out, layout, (reinterpret_cast<uintptr_t>(out) & 31) == 0};
    allow_smem<k_fix_apply>(kFixSmem);
    const int sites = op.parity < 0 ? F.g.vol : F.g.vol / 2, tiles = (sites + 31) / 32;
    k_fix_apply<<<dim3(tiles, fix_grid_y(tiles, n)), kFixThreads, kFixSmem, s>>>(F, op, st, n);
    SEEDCG_CHECK_LAUNCH();
}

// half[h] = full at the parity-p site of h (scatter = 0) or the reverse (scatter = 1), field blockIdx.y
__global__ void k_eo_move(Geom g, int p, int scatter, double2* __restrict__ full, double2* __restrict__ half) {
    const int vh = g.vol / 2;
    const int h = blockIdx.x * blockDim.x + threadIdx.x;
    if (h >= vh) return;
    full += (size_t)blockIdx.y * 12 * g.vol;
    half += (size_t)blockIdx.y * 12 * vh;
    const int s = eo_site(g, h, p);
#pragma unroll
    for (int k = 0; k < 12; k++) {
        if (scatter)
            full[sidx(k, s, g.vol)] = half[sidx(k, h, vh)];
        else
            half[sidx(k, h, vh)] = full[sidx(k, s, g.vol)];
    }
}

void eo_move(const Geom& g, int p, int scatter, int n, double2* full, double2* half, cudaStream_t st) {
    for (int r0 = 0; r0 < n; r0 += kMaxGridY) {
        const dim3 grid((g.vol / 2 + 127) / 128, std::min(n - r0, kMaxGridY));
        k_eo_move<<<grid, 128, 0, st>>>(g, p, scatter, full + (size_t)r0 * 12 * g.vol, half + (size_t)r0 * 6 * g.vol);
        SEEDCG_CHECK_LAUNCH();
    }
}

}  // namespace

void fix_scale(const Geom& g, const double2* u, double kappa, int* k, int* ok, cudaStream_t s) {
    DevBuf rb;
    rb.ensure(2 * sizeof(unsigned));
    unsigned range[2] = {0u, 0x7fffffffu};
    SEEDCG_CUDA_TRY(cudaMemcpyAsync(rb.p, range, sizeof(range), cudaMemcpyHostToDevice, s));
    k_fix_range<<<(4 * g.vol + 255) / 256, 256, 0, s>>>(u, g.vol, rb.as<unsigned>());
    SEEDCG_CHECK_LAUNCH();
    SEEDCG_CUDA_TRY(cudaMemcpyAsync(range, rb.p, sizeof(range), cudaMemcpyDeviceToHost, s));
    SEEDCG_CUDA_TRY(cudaStreamSynchronize(s));
    // |kappa U| < 2^ex for every component, and L = kappa U 2^k stays within 2^55: the exponents are added, as the
    // product need not be a normal number.  Plain FP64 takes links whose largest components are more than 2.5 apart
    // (those of SU(3) links lie between 0.408 = 1 / sqrt(6) and 1): a link is held to 2^-56 of the largest, and next to
    // a point source a hop over links of 1, 1/2, 1/4 of it has an error of 0.88, 1.33, 2.40 times 2^-53 against the
    // chain's 1.06.  It also takes scales so far from the diagonal term's that one of the two, or the factor
    // kappa 2^k, could leave the range.
    *ok = 0;
    *k = 55;
    if (range[0] < 0x7ff00000u - 1u && std::isfinite(kappa)) {
        if (range[0] == 0 || kappa == 0.0) {
            *ok = 1;
        } else {
            const unsigned long long bits[2] = {(unsigned long long)(range[0] + 1u) << 32, (unsigned long long)range[1] << 32};
            double mx = 0.0, mn = 0.0;
            std::memcpy(&mx, &bits[0], sizeof(mx));
            std::memcpy(&mn, &bits[1], sizeof(mn));
            int em = 0, ek = 0, e = 0;
            const double fm = frexp(mx, &em), fk = frexp(std::fabs(kappa), &ek);
            frexp(fm * fk, &e);
            const int ex = em + ek + e;
            *k = 55 - ex;
            *ok = ex >= -100 && ex < 16 && std::abs(ek) <= 500 && std::abs(em) <= 500 && mx <= 2.5 * mn;
        }
    }
}

void fix_links(const Geom& g, const double2* u, double kappa, int k, int4* L, cudaStream_t s) {
    k_fix_links<<<(int)((36L * g.vol + 255) / 256), 256, 0, s>>>(g, u, kappa, k, L);
    SEEDCG_CHECK_LAUNCH();
}

namespace {
void fix_d(const FixDev& F, int dag, int n, const FixView& in, double2* out, const FixView& layout, cudaStream_t s) {
    fix_go(F, FixOp{dag, -1, in, 1, 1, in}, out, layout, n, s);
}

// With t = -kappa H_eo x (FP64 half vectors), A x = x - (-kappa H_oe) t: the factors of
// kappa^2 are in the links.
void fix_a(const FixDev& F, int dag, int n, const FixView& x, double2* te, double2* out, const FixView& layout,
           cudaStream_t st) {
    const FixView t = fix_planes(te, F.g, 1);
    fix_go(F, FixOp{dag, 0, x, 0, 1, x}, te, t, n, st);
    fix_go(F, FixOp{dag, 1, t, 1, -1, x}, out, layout, n, st);
}
}  // namespace

void dslash_f64(const FixDev& F, int dag, int n, const double2* in, double2* out, cudaStream_t s) {
    fix_d(F, dag, n, fix_planes(in, F.g, 0), out, fix_planes(out, F.g, 0), s);
}

void apply_spinors_f64(const FixDev& F, int op, int n, const double* in, double* out, double2* tmp, cudaStream_t s) {
    const double2* x = reinterpret_cast<const double2*>(in);
    double2* y = reinterpret_cast<double2*>(out);
    const FixView vx = fix_spinors(x, F.g, 0), vy = fix_spinors(y, F.g, 0), vt = fix_planes(tmp, F.g, 0);
    if (op < 2) {
        fix_d(F, op, n, vx, y, vy, s);
    } else {
        fix_d(F, 0, n, vx, tmp, vt, s);
        fix_d(F, 1, n, vt, y, vy, s);
    }
}

void apply_eo_spinors_f64(const FixDev& F, int op, int n, const double* in, double* out, double2* te, double2* tmp,
                          cudaStream_t s) {
    const double2* x = reinterpret_cast<const double2*>(in);
    double2* y = reinterpret_cast<double2*>(out);
    const FixView vx = fix_spinors(x, F.g, 1), vy = fix_spinors(y, F.g, 1), vt = fix_planes(tmp, F.g, 1);
    if (op < 2) {
        fix_a(F, op, n, vx, te, y, vy, s);
    } else {
        fix_a(F, 0, n, vx, te, tmp, vt, s);
        fix_a(F, 1, n, vt, te, y, vy, s);
    }
}

void eo_apply_a_f64(const FixDev& F, int dag, int n, const double2* x, double2* te, double2* out, cudaStream_t st) {
    fix_a(F, dag, n, fix_planes(x, F.g, 1), te, out, fix_planes(out, F.g, 1), st);
}

void eo_apply_mdag_m_f64(const FixDev& F, int n, const double2* x, double2* te, double2* out, cudaStream_t st) {
    eo_apply_a_f64(F, 0, n, x, te, out, st);
    eo_apply_a_f64(F, 1, n, out, te, out, st);
}

void eo_source_f64(const FixDev& F, int n, const double2* eta, double2* phi, cudaStream_t st) {
    const FixView v = fix_planes(eta, F.g, 0);
    fix_go(F, FixOp{0, 1, v, 1, -1, v}, phi, fix_planes(phi, F.g, 1), n, st);
}

void eo_gather_f64(const Geom& g, int p, int n, const double2* full, double2* half, cudaStream_t st) {
    eo_move(g, p, 0, n, const_cast<double2*>(full), half, st);
}

void eo_reconstruct_f64(const FixDev& F, int n, const double2* x_odd, const double2* eta, double2* x,
                        cudaStream_t st) {
    fix_go(F, FixOp{0, 0, fix_planes(x_odd, F.g, 1), 1, -1, fix_planes(eta, F.g, 0)}, x, fix_planes(x, F.g, 0), n, st);
    eo_move(F.g, 1, 1, n, x, const_cast<double2*>(x_odd), st);
}

}  // namespace seedcg
