// Even-odd (red-black) preconditioning of the Wilson operator, the setup the
// paper solves (Section 3).  With the sites split by parity (x + y + z + t even
// or odd), D = [[1, -kappa H_eo], [-kappa H_oe, 1]], and eliminating the even
// sites leaves the odd-site Schur complement
//
//     A = 1 - kappa^2 H_oe H_eo,   A x_o = phi = eta_o + kappa H_oe eta_e,
//
// after which x_e = eta_e + kappa H_eo x_o.  A^dag = gamma5 A gamma5 uses the
// hops of D^dag.  A half-lattice vector holds the sites of one parity in
// lexicographic order; with every extent even, half index h and full site s
// satisfy h = s >> 1, because each pair of sites (2h, 2h + 1) holds one site of
// each parity.  Half vectors use the same internal spinor layout as full ones,
// with V/2 sites.
#include <algorithm>
#include <type_traits>

#include "handle.cuh"
#include "internal.cuh"
#include "eo.cuh"
#include "kernels.cuh"
#include "wilson.cuh"

namespace seedcg {
namespace {

constexpr int EOT = 32;   // half sites per block (a lane each); a warp per field, up to 12 side by side

// out[h] = c_diag same[h] + c_hop (H other)(x), x the parity-p_out site of h, for n fields; H is the hopping
// term of D = 1 - kappa H (DAG: of D^dag), `other` the opposite parity.  The tile's links are staged
// once in shared memory for all fields: one field per launch reread them (6.8 us per
// field and hop on 12^3 x 24, 41 us for six; here 21 us).
template <int DAG, typename Out>
__global__ void __launch_bounds__(EOT * 12, 2)
k_eo_hop(Geom g, const float2* __restrict__ u, int p_out, int n, const float2* other,
         const float2* same, float c_diag, float c_hop, Out out) {
    pdl_enter();
    __shared__ float2 sl[2][4][9][EOT];
    __shared__ Nbr snb[EOT];
    __shared__ int ssite[EOT];
    const int vol = g.vol, vh = g.vol / 2;
    const int h0 = blockIdx.x * EOT;
    if (threadIdx.x < EOT && h0 + threadIdx.x < vh) {
        const int s = eo_site(g, h0 + threadIdx.x, p_out);
        ssite[threadIdx.x] = s;
        snb[threadIdx.x] = neighbours(g, s);
    }
    __syncthreads();
    for (int e = threadIdx.x; e < 72 * EOT; e += blockDim.x) {
        const int j = e % EOT, c = (e / EOT) % 9, mu = (e / (9 * EOT)) % 4, dir = e / (36 * EOT);
        if (h0 + j < vh)
            sl[dir][mu][c][j] = __ldg(u + (size_t)(mu * 9 + c) * vol + (dir ? snb[j].b[mu] : ssite[j]));
    }
    __syncthreads();
    const int j = threadIdx.x % EOT, h = h0 + j;
    if (h >= vh) return;
    const Nbr& nb = snb[j];
    auto fl = [&](int mu, int e) { return sl[0][mu][e][j]; };
    auto bl = [&](int mu, int e) { return sl[1][mu][e][j]; };
    const size_t hf = (size_t)vh * 12;
    for (int r = blockIdx.y * (blockDim.x / EOT) + threadIdx.x / EOT; r < n; r += gridDim.y * (blockDim.x / EOT)) {
        links_stay_shared();
        Spinor<float> acc;
        if (same) {
            load_spinor(same + r * hf, vh, h, acc);
#pragma unroll
            for (int k = 0; k < 12; k++) acc.c[k / 3][k % 3] = cscale(acc.c[k / 3][k % 3], c_diag);
        } else {
#pragma unroll
            for (int k = 0; k < 12; k++) acc.c[k / 3][k % 3] = make_float2(0.f, 0.f);
        }
        eo_hops<float, DAG>(nb, fl, bl, other + r * hf, vh, c_hop, acc);
        if constexpr (std::is_same<Out, OutF64>::value) put_spinor_f64(out, (size_t)r * vh + h, acc);
        else store_spinor(out.p + r * hf, vh, h, acc);
    }
}

template <typename Out>
void eo_hop(const Geom& g, const float2* u, int dag, int p_out, int n, const float2* other, const float2* same,
            float c_diag, float c_hop, Out out, cudaStream_t st) {
    const int tiles = (g.vol / 2 + EOT - 1) / EOT;
    // fields side by side: all of them in balanced passes of at most 12 warps, split over the grid while the
    // tiles alone do not fill two blocks per SM
    const int gy = std::min({n, kMaxGridY, std::max((n + 11) / 12, (304 + tiles - 1) / tiles)});
    const int per = std::min(12, (n + gy - 1) / gy);
    launch_pdl(pdl_for_apply(6L * g.vol * n), dag ? k_eo_hop<1, Out> : k_eo_hop<0, Out>, dim3(tiles, gy), EOT * per, 0,
               st, g, u, p_out, n, other, same, c_diag, c_hop, out);
}

// y_o = A x_o (dag = 0) or A^dag x_o (dag = 1), n half vectors; t: even-site scratch
template <typename Out>
void apply_a(const Geom& g, const float2* u, double kappa, int dag, int n, const float2* x, float2* t, Out y,
             cudaStream_t st) {
    eo_hop(g, u, dag, 0, n, x, nullptr, 0.f, 1.f, OutF32{t}, st);                        // H_eo x
    eo_hop(g, u, dag, 1, n, t, x, 1.f, (float)(-kappa * kappa), y, st);                  // x - k^2 H_oe t
}

}  // namespace

namespace {

bool eo_dims_ok(const Geom& g) {
    for (int mu = 0; mu < 4; mu++)
        if (g.L[mu] % 2) return false;
    return true;
}

void apply_eo_f64(seedcg_handle* h, int op, int n, const double* in, double* out, cudaStream_t st) {
    const size_t hf = (size_t)h->g.vol / 2 * 12 * n;
    KeptScratch::Use work(h->apply, (op == 2 ? 2 : 1) * hf * sizeof(double2));
    double2* te = work.as<double2>();
    apply_eo_spinors_f64(fix_of(h), op, n, in, out, te, te + hf, st);
    SEEDCG_CUDA_TRY(cudaStreamSynchronize(st));
}

void apply_eo_f32(seedcg_handle* h, int op, int n, const double* in, double* out, cudaStream_t st) {
    const size_t hf = (size_t)h->g.vol / 2 * 12 * n;
    KeptScratch::Use work(h->apply, (op == 2 ? 3 : 2) * hf * sizeof(float2));
    const float2* u = h->u32.as<float2>();
    float2* X = work.as<float2>();
    float2* T = X + hf;
    float2* Y = T + hf;   // op 2 only
    to_internal_f32(in, X, h->g.vol / 2, n, st);
    if (op < 2) {
        apply_a(h->g, u, h->kappa, op, n, X, T, make_out_f64(out), st);
    } else {
        apply_a(h->g, u, h->kappa, 0, n, X, T, OutF32{Y}, st);
        apply_a(h->g, u, h->kappa, 1, n, Y, T, make_out_f64(out), st);
    }
    SEEDCG_CUDA_TRY(cudaStreamSynchronize(st));
}

bool is_dev(const void* p) {
    cudaPointerAttributes a;
    if (cudaPointerGetAttributes(&a, p) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    return a.type == cudaMemoryTypeDevice || a.type == cudaMemoryTypeManaged;
}

seedcg_status check_eo(seedcg_handle* h, int n, std::initializer_list<const void*> ptrs) {
    if (!h) return SEEDCG_ERR_ARG;
    if (n < 1) {
        h->err = "n must be >= 1";
        return SEEDCG_ERR_ARG;
    }
    if (!eo_dims_ok(h->g)) {
        h->err = "even-odd preconditioning needs every lattice extent even";
        return SEEDCG_ERR_ARG;
    }
    for (const void* p : ptrs)
        if (!p || !is_dev(p)) {
            h->err = "even-odd calls take device pointers";
            return SEEDCG_ERR_ARG;
        }
    return SEEDCG_OK;
}

}  // namespace
}  // namespace seedcg

using seedcg::DevBuf;
using seedcg::Error;

extern "C" seedcg_status seedcg_apply_eo(seedcg_handle* h, int op, int prec, int n, const double* in,
                                         double* out, void* stream) {
    seedcg_status c = seedcg::check_eo(h, n, {in, out});
    if (c != SEEDCG_OK) return c;
    if (op < 0 || op > 2 || prec < 0 || prec > 1 || in == out) {
        h->err = "bad op / prec, or in and out alias";
        return SEEDCG_ERR_ARG;
    }
    try {
        SEEDCG_CUDA_TRY(cudaSetDevice(h->device));
        cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
        if (prec == 0) seedcg::apply_eo_f64(h, op, n, in, out, st);
        else seedcg::apply_eo_f32(h, op, n, in, out, st);
        return SEEDCG_OK;
    } catch (const Error& e) {
        h->err = e.msg;
        return e.code;
    }
}

extern "C" seedcg_status seedcg_eo_source(seedcg_handle* h, int n, const double* eta, double* phi,
                                          void* stream) {
    seedcg_status c = seedcg::check_eo(h, n, {eta, phi});
    if (c != SEEDCG_OK) return c;
    try {
        SEEDCG_CUDA_TRY(cudaSetDevice(h->device));
        cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
        const seedcg::Geom& g = h->g;
        const int vh = g.vol / 2;
        const size_t hf = (size_t)vh * 12, ff = (size_t)g.vol * 12;
        DevBuf buf;
        buf.ensure(((size_t)n * ff + (size_t)n * hf) * sizeof(double2));
        double2* E = buf.as<double2>();
        double2* P = E + (size_t)n * ff;
        seedcg::to_internal_f64(eta, E, g.vol, n, st);
        seedcg::eo_source_f64(seedcg::fix_of(h), n, E, P, st);   // phi = eta_o + kappa H_oe eta_e
        seedcg::from_internal_f64(P, phi, vh, n, st);
        SEEDCG_CUDA_TRY(cudaStreamSynchronize(st));
        return SEEDCG_OK;
    } catch (const Error& e) {
        h->err = e.msg;
        return e.code;
    }
}

extern "C" seedcg_status seedcg_eo_reconstruct(seedcg_handle* h, int n, const double* x_odd,
                                               const double* eta, double* x, void* stream) {
    seedcg_status c = seedcg::check_eo(h, n, {x_odd, eta, x});
    if (c != SEEDCG_OK) return c;
    try {
        SEEDCG_CUDA_TRY(cudaSetDevice(h->device));
        cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
        const seedcg::Geom& g = h->g;
        const int vh = g.vol / 2;
        const size_t hf = (size_t)vh * 12, ff = (size_t)g.vol * 12;
        DevBuf buf;
        buf.ensure((2 * (size_t)n * ff + (size_t)n * hf) * sizeof(double2));
        double2* E = buf.as<double2>();
        double2* F = E + (size_t)n * ff;
        double2* Xo = F + (size_t)n * ff;
        seedcg::to_internal_f64(eta, E, g.vol, n, st);
        seedcg::to_internal_f64(x_odd, Xo, vh, n, st);
        seedcg::eo_reconstruct_f64(seedcg::fix_of(h), n, Xo, E, F, st);   // x_e = eta_e + kappa H_eo x_o
        seedcg::from_internal_f64(F, x, g.vol, n, st);
        SEEDCG_CUDA_TRY(cudaStreamSynchronize(st));
        return SEEDCG_OK;
    } catch (const Error& e) {
        h->err = e.msg;
        return e.code;
    }
}

extern "C" seedcg_status seedcg_solve_eo(seedcg_handle* h, int nrhs, const double* eta, double* x, double tol,
                                         int extra_iters, int reorth_period, seedcg_info* info, void* stream) {
    seedcg_status c = seedcg::check_eo(h, nrhs, {eta, x});
    if (c != SEEDCG_OK) return c;
    if (!(tol > 0.0) || !(tol < 1.0) || extra_iters < 0 || reorth_period < 0 || nrhs > 256 || eta == x) {
        h->err = "bad tol, extra_iters, reorth_period or nrhs, or eta and x alias";
        return SEEDCG_ERR_ARG;
    }
    if (h->opt.use_guess || h->opt.resid_mode != 0) {
        h->err = "seedcg_solve_eo: use_guess and resid_mode = 1 are full-lattice options (the original "
                 "system's residual is reported in info->true_resid_D)";
        return SEEDCG_ERR_ARG;
    }
    try {
        SEEDCG_CUDA_TRY(cudaSetDevice(h->device));
        return seedcg::solve_eo_impl(h, nrhs, eta, x, tol, extra_iters, reorth_period, info,
                                     reinterpret_cast<cudaStream_t>(stream));
    } catch (const Error& e) {
        h->err = e.msg;
        return e.code;
    }
}
