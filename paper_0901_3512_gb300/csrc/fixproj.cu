// The FP64 basis products of fixproj.cuh: V^dag X for a few vectors and Y += V C.
#include <algorithm>

#include "fixproj.cuh"

namespace seedcg {
namespace {

// Block (x, y): a chunk of entries against the rows of group y, like k_proj_partial: the chunk of X in shared memory
// as limbs, a warp takes RPW rows at a time, a lane every 32nd entry.  A lane adds at most 16 entries (32
// products of at most 2^56), so 64 bits hold its sums; the warp's sum is formed exactly from three 22-bit
// parts.  RPW * NV * 2 values per warp are converted to FP64 side by side.  8^3 x 16, 320 rows on average, two
// vectors: 570 us on the FP64 pipe, 160 us here (issue-bound; the rows take 75 us at the measured HBM rate); eleven
// seed vectors against 634 rows: 5.1 -> 1.6 ms, and their X += V Y 5.7 -> 1.9 ms.
template <int NV, int RPW, int CHUNK>
__global__ void __launch_bounds__(256, 2)
k_proj_fix(const double2* V, long ldv, int na, const int* runE,
           const double2* X, long ldx, int nv, long n, int chunk, int rg, double2* __restrict__ part) {
    static_assert(RPW * NV * 2 <= 32, "one lane per value");
    pdl_enter();
    __shared__ int4 sx[NV][CHUNK];
    __shared__ int s_mx[NV + 1];
    const long e0 = (long)blockIdx.x * chunk;
    const int cnt = (int)(n - e0 < chunk ? n - e0 : chunk);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
    if (threadIdx.x <= NV) s_mx[threadIdx.x] = kFixEMin << 20;
    __syncthreads();
#pragma unroll
    for (int j = 0; j < NV; j++) {
        int m = 0;
        if (j < nv)
            for (int e = threadIdx.x; e < cnt; e += blockDim.x) m = max(m, fix_absword(X[(size_t)j * ldx + e0 + e]));
        m = __reduce_max_sync(0xffffffffu, m);
        if (lane == 0) atomicMax(&s_mx[j], m);
    }
    {
        int m = 0;
        for (int b = threadIdx.x; b < cnt / kFixBlock; b += blockDim.x) m = max(m, runE[e0 / kFixBlock + b]);
        m = __reduce_max_sync(0xffffffffu, m);
        if (lane == 0) atomicMax(&s_mx[NV], m << 20);
    }
    __syncthreads();
    for (int k = threadIdx.x; k < NV * cnt; k += blockDim.x) {
        const int j = k / cnt, e = k % cnt;
        const double2 z = j < nv ? X[(size_t)j * ldx + e0 + e] : make_double2(0.0, 0.0);
        const int eb = s_mx[j] & 0x7ff00000;
        int4 w;
        fix_limbs(z.x, eb, 0u, w.x, w.y);
        fix_limbs(z.y, eb, 0u, w.z, w.w);
        sx[j][e] = w;
    }
    __syncthreads();
    const int Ev = s_mx[NV] >> 20, vb = Ev << 20;
    double2* out = part + (size_t)blockIdx.x * na * NV;
    const int rbeg = blockIdx.y * rg, rend = rbeg + rg < na ? rbeg + rg : na;
    for (int a0 = rbeg + warp * RPW; a0 < rend; a0 += nw * RPW) {
        long long A[RPW][NV][2], B[RPW][NV][2];
#pragma unroll
        for (int r = 0; r < RPW; r++)
#pragma unroll
            for (int j = 0; j < NV; j++) A[r][j][0] = A[r][j][1] = B[r][j][0] = B[r][j][1] = 0;
        const double2* rows[RPW];
#pragma unroll
        for (int r = 0; r < RPW; r++) rows[r] = V + (size_t)(a0 + r < rend ? a0 + r : a0) * ldv + e0;
#pragma unroll 2
        for (int e = lane; e < cnt; e += 32) {
            double2 z[RPW];
#pragma unroll
            for (int r = 0; r < RPW; r++) z[r] = __ldcs(rows[r] + e);
            int4 x[NV];
#pragma unroll
            for (int j = 0; j < NV; j++) x[j] = sx[j][e];
#pragma unroll
            for (int r = 0; r < RPW; r++) {
                int rh, rl, ih, il;
                fix_limbs(z[r].x, vb, 0u, rh, rl);
                fix_limbs(z[r].y, vb, 0u, ih, il);
                const int nh = -ih, nl = -il;
#pragma unroll
                for (int j = 0; j < NV; j++) {
                    // conj(v) x
                    A[r][j][0] += (long long)rh * x[j].x;
                    B[r][j][0] += (long long)rh * x[j].y;
                    B[r][j][0] += (long long)rl * x[j].x;
                    A[r][j][0] += (long long)ih * x[j].z;
                    B[r][j][0] += (long long)ih * x[j].w;
                    B[r][j][0] += (long long)il * x[j].z;
                    A[r][j][1] += (long long)rh * x[j].z;
                    B[r][j][1] += (long long)rh * x[j].w;
                    B[r][j][1] += (long long)rl * x[j].z;
                    A[r][j][1] += (long long)nh * x[j].x;
                    B[r][j][1] += (long long)nh * x[j].y;
                    B[r][j][1] += (long long)nl * x[j].x;
                }
            }
        }
        // the warp's exact sums, value k = (r * NV + j) * 2 + part kept by lane k
        long long mine = 0;
        int drop = 0;
#pragma unroll
        for (int r = 0; r < RPW; r++)
#pragma unroll
            for (int j = 0; j < NV; j++)
#pragma unroll
                for (int q = 0; q < 2; q++) {
                    const long long t = A[r][j][q] + (B[r][j][q] >> 27);
                    const unsigned s0 = __reduce_add_sync(0xffffffffu, (unsigned)t & 0x3fffffu);
                    const unsigned s1 = __reduce_add_sync(0xffffffffu, (unsigned)(t >> 22) & 0x3fffffu);
                    const int s2 = __reduce_add_sync(0xffffffffu, (int)(t >> 44));
                    if (lane == (r * NV + j) * 2 + q) {
                        const long long hi = ((long long)s2 << 22) + s1;
                        const bool big = hi >= (1ll << 40) || hi < -(1ll << 40);
                        drop = big ? 8 : 0;
                        mine = big ? (hi << 14) + (s0 >> 8) : (hi << 22) + s0;
                    }
                }
        if (lane < RPW * NV * 2) {
            const int q = lane & 1, j = (lane >> 1) % NV, r = (lane >> 1) / NV;
            const int Ex = s_mx[j] >> 20;
            const bool bad = Ev > kFixEMax || Ex > kFixEMax;
            const double d = bad ? __longlong_as_double(0x7ff8000000000000ll) : ldexp((double)mine, Ev + Ex - 2100 + drop);
            if (a0 + r < rend && j < nv) reinterpret_cast<double*>(out)[((size_t)(a0 + r) * NV + j) * 2 + q] = d;
        }
    }
}

// C[a][j] = sum over blocks of part[b][a][j]: one warp per output, fixed order
template <int NV>
__global__ void k_proj_fix_reduce(const double2* part, int nblk, int na, int nv, double2* __restrict__ C,
                                  int ldc, int c0) {
    pdl_enter();
    const int w = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int lane = threadIdx.x & 31;
    if (w >= na * nv) return;
    const int a = w / nv, j = w % nv;
    double re = 0.0, im = 0.0;
    for (int b = lane; b < nblk; b += 32) {
        const double2 z = part[((size_t)b * na + a) * NV + j];
        re += z.x;
        im += z.y;
    }
    re = warp_sum(re);
    im = warp_sum(im);
    if (lane == 0) C[(size_t)a * ldc + c0 + j] = make_double2(re, im);
}

constexpr int kChunk = 512;   // entries staged per block at most (NV = 4: 32 KB)

// enough blocks to fill the SMs twice; whole exponent blocks and whole warps of entries
inline int chunk_for(long n) {
    long c = (n + 303) / 304;
    c = (c + 31) / 32 * 32;
    return (int)std::min<long>(std::max<long>(c, 64), kChunk);
}

template <int NV, int RPW>
void proj_pass(const double2* V, long ldv, int na, const int* runE, const double2* X, long ldx, int nv, long n,
               double2* C, int ldc, int c0, double2* scratch, cudaStream_t s) {
    const int ch = chunk_for(n);
    const int nblk = (int)((n + ch - 1) / ch);
    // rows per block: two trips per warp, fewer when the chunks alone do not fill the chip
    const int per = 8 * RPW;
    const int want = std::max(1, (4 * 152 + nblk - 1) / nblk);
    const int rg = std::max(per, std::min((na + want - 1) / want, 16 * per) / per * per);
    launch_pdl(pdl_for(n), k_proj_fix<NV, RPW, kChunk>, dim3(nblk, (na + rg - 1) / rg), 256, 0, s, V, ldv, na, runE, X,
               ldx, nv, n, ch, rg, scratch);
    launch_pdl(pdl_for(n), k_proj_fix_reduce<NV>, (na * nv + 7) / 8, 256, 0, s, scratch, nblk, na, nv, C, ldc, c0);
}

template <int NB>
__global__ void __launch_bounds__(256, 2)
k_gemm_n_fix(const double2* __restrict__ V, long ldv, int na, const int* __restrict__ runE,
             const double2* __restrict__ C, int ldc, int nb, int b0, double2* __restrict__ Y, long ldy, long n) {
    __shared__ FixColumns<NB> S;
    const long e = blockIdx.x * (long)blockDim.x + threadIdx.x;
    int col[NB];
#pragma unroll
    for (int j = 0; j < NB; j++) col[j] = b0 + j < nb ? b0 + j : -1;
    double2 av[NB];
    fix_accumulate<NB>(V, ldv, 0, na, runE, C, ldc, col, e, e < n, av, S);
    if (e >= n) return;
#pragma unroll
    for (int j = 0; j < NB; j++)
        if (col[j] >= 0) {
            double2 y = Y[(size_t)(b0 + j) * ldy + e];
            y.x += av[j].x;
            y.y += av[j].y;
            Y[(size_t)(b0 + j) * ldy + e] = y;
        }
}

}  // namespace

size_t proj_fix_scratch(long n, int na) { return (size_t)((n + chunk_for(n) - 1) / chunk_for(n)) * 2 * na; }

void proj_fix(const double2* V, long ldv, int na, const int* runE, const double2* X, long ldx, int nx, long n,
              double2* C, int ldc, double2* scratch, size_t scratch_elems, cudaStream_t s) {
    if (na <= 0 || nx <= 0) return;
    if (n % 32 != 0 || proj_fix_scratch(n, na) > scratch_elems) throw Error{SEEDCG_ERR_OOM, "proj scratch"};
    // two vectors (the re-orthogonalisation) or, when the partials fit, four (the seeds) per pass over V
    const int most = 2 * proj_fix_scratch(n, na) <= scratch_elems ? 4 : 2;
    for (int c0 = 0; c0 < nx;) {
        const int nv = std::min(most, nx - c0);
        const double2* Xc = X + (size_t)c0 * ldx;
        if (nv <= 2) proj_pass<2, 4>(V, ldv, na, runE, Xc, ldx, nv, n, C, ldc, c0, scratch, s);
        else proj_pass<4, 2>(V, ldv, na, runE, Xc, ldx, nv, n, C, ldc, c0, scratch, s);
        c0 += nv;
    }
}

void gemm_n_fix(const double2* V, long ldv, int na, const int* runE, const double2* C, int ldc, int nb, double2* Y,
                long ldy, long n, cudaStream_t s) {
    if (na <= 0 || nb <= 0 || n <= 0) return;
    for (int b0 = 0; b0 < nb; b0 += 4) {
        k_gemm_n_fix<4><<<(int)((n + 255) / 256), 256, 0, s>>>(V, ldv, na, runE, C, ldc, nb, b0, Y, ldy, n);
        SEEDCG_CHECK_LAUNCH();
    }
}

}  // namespace seedcg
