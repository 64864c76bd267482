// Products with the stored FP64 basis V in fixed point on the integer pipe (as fixhop.cuh; an FP64
// multiply-add is 40 times rarer than a 32 x 32 + 64 bit one on this GPU).
//
// An entry of V is taken relative to E(block), the largest exponent that any stored row has among the 16 entries of its
// block (a running maximum kept while rows are stored, fix_row_exponent), a vector or coefficient relative to
// its largest component in the chunk or column.  Every product is exact up to its lowest 2^-57,
// sums are exact, and a sum becomes FP64 once per (row, chunk) or (entry, segment).  The error of an inner
// product is about 2^-56 max|v| ||x|| sqrt(1/32 .. 1), against 2^-54 |partial sum| per addition in FP64.
#pragma once

#include "fixhop.cuh"

namespace seedcg {

constexpr int kFixBlock = 16;   // entries per exponent; every vector length is a multiple (12 * 8 sites or more)

// row[e]'s contribution to the running exponents: threads of 16 / W consecutive lanes hold a block (W entries each);
// `h` is the largest upper word (sign cleared) among the thread's components.  Every lane of the group calls it.
template <int W>
__device__ __forceinline__ void fix_row_exponent(int* runE, long e, int h, unsigned mask) {
#pragma unroll
    for (int o = kFixBlock / W / 2; o > 0; o >>= 1) h = max(h, __shfl_xor_sync(mask, h, o));
    if (e % kFixBlock == 0) {
        const int b = (int)(e / kFixBlock);
        runE[b] = max(runE[b], h >> 20);
    }
}
__device__ __forceinline__ int fix_absword(double2 z) {
    return max(__double2hiint(z.x) & 0x7fffffff, __double2hiint(z.y) & 0x7fffffff);
}

// C[a][j] = sum_e conj(V[a][e]) X[j][e], a < na, j < nx (scratch: proj_fix_scratch elements)
size_t proj_fix_scratch(long n, int na);
void proj_fix(const double2* V, long ldv, int na, const int* runE, const double2* X, long ldx, int nx, long n,
              double2* C, int ldc, double2* scratch, size_t scratch_elems, cudaStream_t s);
// Y[j][e] += sum_a V[a][e] C[a][j], j < nb
void gemm_n_fix(const double2* V, long ldv, int na, const int* runE, const double2* C, int ldc, int nb, double2* Y,
                long ldy, long n, cudaStream_t s);

// Sums of V[a][e] c[a][j] over rows for one entry e per thread, NB columns: limbs of 64 rows' coefficients at a time
// in shared memory; 32 rows of products fit 64 bits, longer sums 96.
template <int NB>
struct FixColumns {
    static constexpr int CH = 64;
    int4 c[CH][NB];
    int ebits[NB];   // exponent field of each column's coefficients
    int red[8][NB];
};

// av[j] = sum over rows [r0, r1) of V[a][e] coef[a * ldc + col[j]]; every thread of the block (256) calls it
template <int NB>
__device__ __forceinline__ void fix_accumulate(const double2* V, long ldv, int r0, int r1,
                                               const int* runE, const double2* coef, int ldc,
                                               const int (&col)[NB], long e, bool live, double2 (&av)[NB],
                                               FixColumns<NB>& S) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // the columns' exponents over these rows
    {
        int mx[NB];
#pragma unroll
        for (int j = 0; j < NB; j++) mx[j] = 0;
        for (int a = r0 + threadIdx.x; a < r1; a += blockDim.x)
#pragma unroll
            for (int j = 0; j < NB; j++) mx[j] = max(mx[j], col[j] >= 0 ? fix_absword(coef[(size_t)a * ldc + col[j]]) : 0);
#pragma unroll
        for (int j = 0; j < NB; j++) {
            mx[j] = __reduce_max_sync(0xffffffffu, mx[j]);
            if (lane == 0) S.red[warp][j] = mx[j];
        }
        __syncthreads();
        if (threadIdx.x < NB) {
            int m = 0;
            for (int w = 0; w < (int)(blockDim.x >> 5); w++) m = max(m, S.red[w][threadIdx.x]);
            S.ebits[threadIdx.x] = max(m >> 20, kFixEMin) << 20;
        }
    }
    const int Ev = live ? max(runE[e / kFixBlock], kFixEMin) : kFixEMin;
    const int vb = Ev << 20;
    long long lo[2 * NB];
    int hi[2 * NB];
#pragma unroll
    for (int k = 0; k < 2 * NB; k++) {
        lo[k] = 0;
        hi[k] = 0;
    }
    constexpr int CH = FixColumns<NB>::CH;
    for (int a0 = r0; a0 < r1; a0 += CH) {
        const int cnt = min(CH, r1 - a0);
        __syncthreads();
        for (int k = threadIdx.x; k < CH * NB; k += blockDim.x) {
            const int a = k / NB, j = k % NB;
            int cj = -1;
#pragma unroll
            for (int q = 0; q < NB; q++)
                if (q == j) cj = col[q];
            const double2 z = a < cnt && cj >= 0 ? coef[(size_t)(a0 + a) * ldc + cj] : make_double2(0.0, 0.0);
            int4 w;
            fix_limbs(z.x, S.ebits[j], 0u, w.x, w.y);
            fix_limbs(z.y, S.ebits[j], 0u, w.z, w.w);
            S.c[a][j] = w;
        }
        __syncthreads();
        if (!live) continue;
        for (int h0 = 0; h0 < cnt; h0 += 32) {
            long long A[2 * NB], B[2 * NB];
#pragma unroll
            for (int k = 0; k < 2 * NB; k++) A[k] = B[k] = 0;
            const int top = min(h0 + 32, cnt);
            const double2* p = V + (size_t)(a0 + h0) * ldv + e;
#pragma unroll 4
            for (int a = h0; a < top; a++, p += ldv) {
                const double2 z = __ldcs(p);
                int rh, rl, ih, il;
                fix_limbs(z.x, vb, 0u, rh, rl);
                fix_limbs(z.y, vb, 0u, ih, il);
                const int nh = -ih, nl = -il;
#pragma unroll
                for (int j = 0; j < NB; j++) {
                    const int4 c = S.c[a][j];
                    A[2 * j] += (long long)rh * c.x;
                    B[2 * j] += (long long)rh * c.y;
                    B[2 * j] += (long long)rl * c.x;
                    A[2 * j] += (long long)nh * c.z;
                    B[2 * j] += (long long)nh * c.w;
                    B[2 * j] += (long long)nl * c.z;
                    A[2 * j + 1] += (long long)rh * c.z;
                    B[2 * j + 1] += (long long)rh * c.w;
                    B[2 * j + 1] += (long long)rl * c.z;
                    A[2 * j + 1] += (long long)ih * c.x;
                    B[2 * j + 1] += (long long)ih * c.y;
                    B[2 * j + 1] += (long long)il * c.x;
                }
            }
#pragma unroll
            for (int k = 0; k < 2 * NB; k++) {
                const long long r = A[k] + (B[k] >> 27), o = lo[k];
                lo[k] = (long long)((unsigned long long)o + (unsigned long long)r);
                hi[k] += (int)(r >> 63) + ((unsigned long long)lo[k] < (unsigned long long)o ? 1 : 0);
            }
        }
    }
    const bool bad = Ev > kFixEMax;
#pragma unroll
    for (int j = 0; j < NB; j++) {
        double v[2];
#pragma unroll
        for (int q = 0; q < 2; q++) {
            const int k = 2 * j + q;
            // 96 bits: the upper word is the sign until products of one sign near the largest fill 64 bits (about 128 rows
            // of them); then as many bits are dropped as the upper word takes, which leaves at least 62
            const bool fits = hi[k] == (int)(lo[k] >> 63);
            const int drop = fits ? 0 : 33 - __clz(hi[k] ^ (hi[k] >> 31));
            const long long t = fits ? lo[k] : (long long)(((unsigned long long)(long long)hi[k] << (64 - drop)) | ((unsigned long long)lo[k] >> drop));
            const int ec = S.ebits[j] >> 20;
            // unit of hi x hi: 2^(54 - 2 * 1077 + Ev + Ec)
            v[q] = bad || ec > kFixEMax ? __longlong_as_double(0x7ff8000000000000ll)
                                        : ldexp((double)t, Ev + ec - 2100 + drop);
        }
        av[j] = make_double2(v[0], v[1]);
    }
}

}  // namespace seedcg
