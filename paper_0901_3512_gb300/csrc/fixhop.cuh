// The FP64 Wilson hopping term in 64-bit fixed point on the integer pipe.
//
// GB300 executes FP64 at 1.6 lanes per clock and SM (a DFMA or DADD occupies an SM
// partition for 68 clocks, measured), against 54 for a 32 x 32 + 64 bit integer
// multiply-add.  A hop's 3 x 3 complex products are therefore formed exactly in
// integers: each half spinor of the projection becomes 12 fixed-point numbers relative to the exponent E of the
// largest component that goes into it (55 fraction bits: one step is 2^-55 of a power of two at
// most twice that component), a link is L = -kappa U 2^k with |L| <= 2^55 (prepared
// once per handle, the antiperiodic sign included), both split into a 27-bit low and
// a 29-bit high limb.  A product needs three 32 x 32 multiply-adds (high x high and the two
// cross terms; low x low is below 2^-57 of the result), sums are exact, and the sums
// of the eight hops are aligned to the largest E among them and added to the
// diagonal term before the one rounding to FP64.  The error is at most a few 2^-55 of the largest
// component among the spins that an output spin takes from the neighbours: below that of the FP64 chain it replaces,
// which rounds about 20 times per component, on dense fields and for each spin.  A single colour far below its
// spin's others counts against those.
//
// One block owns 32 sites and one warp one of the eight directions, so a link stays in
// registers for all right-hand sides of the block; the eight warps meet in shared memory,
// where six of them add the directions up, one pair-plane (two complex entries of
// every site) each.  D on 12 fields at 16^3 x 32: 2489 us with the FP64 chain, 900 us here; one
// field at 8^3 x 16 in the Lanczos loop 31 -> 8.2 us, at 4^4 31 -> 5.5 us.
//
// Sites whose neighbourhood holds values that the fixed point cannot take (infinities, NaN,
// magnitudes beyond 2^+-800) are computed by the plain FP64 chain (fix_chain), and so is every site of a handle whose
// links differ in size by more than 2.5 (ok = 0; never SU(3) links): there a warp takes 32 sites of one field (fix_plain).
#pragma once

#include "eo.cuh"
#include "internal.cuh"
#include "reduce.cuh"
#include "wilson.cuh"

namespace seedcg {

constexpr int kFixThreads = 256;
constexpr int kFixEMin = 200, kFixEMax = 1900;   // biased exponents the fixed point accepts
constexpr int kFixBad = 0x7fffffff;
// two buffers of [8 directions][12 components][32 sites] 64-bit sums and [2 spins][8][32] exponents, the
// six planes' shares per buffer
constexpr size_t kFixBufBytes = 8 * 12 * 32 * sizeof(long long) + 2 * 8 * 32 * sizeof(int);
constexpr size_t kFixSmem = 2 * kFixBufBytes + 2 * 8 * sizeof(double);

// x (a double with sign flipped where flip has bit 31) as two limbs x = (hi 2^27 + lo) 2^(E - 1022 - 55);
// ebits = E << 20, E at least x's exponent.  Bits below the last step are cut off.
__device__ __forceinline__ void fix_limbs(double x, int ebits, unsigned flip, int& hi, int& lo) {
    const unsigned h = (unsigned)__double2hiint(x) ^ flip, l = (unsigned)__double2loint(x);
    const unsigned d = (unsigned)(ebits - (int)(h & 0x7ff00000u)) >> 20;
    const unsigned mh = (h & 0x000fffffu) | 0x00100000u;
    const unsigned MH = __funnelshift_l(l, mh, 11), ML = l << 11;   // 53-bit significand at the top
    unsigned uh, ul;
    asm("shr.u32 %0, %1, %2;" : "=r"(uh) : "r"(MH), "r"(d + 4));    // shifts past 31 give 0
    asm("{ .reg .b64 t; mov.b64 t, {%1, %2}; shr.u64 t, t, %3; cvt.u32.u64 %0, t; }"
        : "=r"(ul) : "r"(ML), "r"(MH), "r"(d + 9));
    ul &= 0x07ffffffu;
    const int s = (int)h >> 31;
    hi = ((int)uh ^ s) - s;
    lo = ((int)ul ^ s) - s;
}

// arithmetic shift right that saturates (a shift of 63 or more leaves the sign)
__device__ __forceinline__ long long fix_sra(long long v, int n) {
    long long r;
    asm("shr.s64 %0, %1, %2;" : "=l"(r) : "l"(v), "r"(n));
    return r;
}

// Sums are integers in units of 2^(-1 - kFixUnit) 2^(E - 1022): E is the neighbours' exponent, moved by the links' scale
// (L = -kappa U 2^k: E + kFixUnit - k), so the unit follows the hop's size whatever kappa is, and every exponent
// below stays a normal one for k in (39, 155].
constexpr int kFixUnit = 57;

// S in that unit, rounded to FP64 (S != 0)
__device__ __forceinline__ double fix_to_double(long long S, int E) {
    const unsigned long long a = S < 0 ? (unsigned long long)(-S) : (unsigned long long)S;
    const int n = __clzll((long long)a);
    const unsigned long long t = a << n;
    const unsigned long long q = (t >> 11) + ((t >> 10) & 1ull);   // 53 bits, rounded half up
    const long long eb = (long long)(E + 63 - n - kFixUnit);
    const unsigned long long bits = ((unsigned long long)(eb - 1) << 52) + q;
    return __longlong_as_double((long long)(bits | (S < 0 ? 0x8000000000000000ull : 0ull)));
}

// diag * p + sgn * S, the diagonal term p in FP64 (diag 0 or 1)
__device__ __forceinline__ double fix_combine(long long S, int E, int diag, double p) {
    if (S == 0) return diag ? p : 0.0;
    if (!diag) return fix_to_double(S, E);
    const unsigned h = (unsigned)__double2hiint(p), l = (unsigned)__double2loint(p);
    const int e = (int)((h >> 20) & 0x7ffu);
    if (e == 0) return fix_to_double(S, E);   // zero, or below every step of S
    const int Ec = e > E ? e : E;
    const unsigned long long m = ((unsigned long long)((h & 0x000fffffu) | 0x00100000u) << 32) | l;
    // p's significand (below 2^53) in the unit of Ec
    const int sh = kFixUnit - 52 - (Ec - e);
    unsigned long long P;
    if (sh >= 0) P = m << sh;
    else asm("shr.u64 %0, %1, %2;" : "=l"(P) : "l"(m), "r"(-sh));
    const long long sp = (int)h < 0 ? -(long long)P : (long long)P;
    const long long T = fix_sra(S, Ec - E) + sp;
    return T == 0 ? 0.0 : fix_to_double(T, Ec);
}

// FP64 fields as the tiles read them: entry k of site y of field r at p[r * field + y * site + (k / 2) * pair + k % 2].
// Internal fields are pair planes (site 2, pair 2 * sites), the boundary's fields spinors (site 12, pair 2), which the
// operator reads and writes in place: no layout pass.  half = 1: half vectors (y is the half index).
struct FixView {
    const double2* p;
    long field;
    int site, pair, half;
};
inline FixView fix_planes(const double2* p, const Geom& g, int half) {
    return FixView{p, 12L * (g.vol >> half), 2, 2 * (g.vol >> half), half};
}
inline FixView fix_spinors(const double2* p, const Geom& g, int half) {
    return FixView{p, 12L * (g.vol >> half), 12, 2, half};
}

// -kappa H psi (dag: of D^dag's hopping term) at full site s, by the plain FP64 chain; psi: field r of `in`
static __device__ __noinline__ void fix_chain(const FixDev& F, int dag, int s, const FixView& in, int r, double2* out) {
    const Geom& g = F.g;
    const Nbr nb = neighbours(g, s);
    const int vol = g.vol, sh = in.half;
    Spinor<double> acc;
#pragma unroll
    for (int k = 0; k < 12; k++) acc.c[k / 3][k % 3] = make_double2(0.0, 0.0);
    auto fl = [&](int mu, int e) { return __ldg(F.u + (size_t)(mu * 9 + e) * vol + s); };
    auto bl = [&](int mu, int e) { return __ldg(F.u + (size_t)(mu * 9 + e) * vol + nb.b[mu]); };
    Nbr idx = nb;
#pragma unroll
    for (int mu = 0; mu < 4; mu++) {
        idx.f[mu] = nb.f[mu] >> sh;
        idx.b[mu] = nb.b[mu] >> sh;
    }
    auto load = [&](int y, Spinor<double>& p) {
        if (y < 0) {   // the diagonal term: none here
#pragma unroll
            for (int k = 0; k < 12; k++) p.c[k / 3][k % 3] = make_double2(0.0, 0.0);
        } else {
            const double2* q = in.p + (size_t)r * in.field + (size_t)y * in.site;
#pragma unroll
            for (int k = 0; k < 12; k++) p.c[k / 3][k % 3] = q[(size_t)(k >> 1) * in.pair + (k & 1)];
        }
    };
    if (dag) wilson_site<1, double>(idx, -1, load, fl, bl, F.kappa, acc);
    else wilson_site<0, double>(idx, -1, load, fl, bl, F.kappa, acc);
#pragma unroll
    for (int k = 0; k < 12; k++) out[k] = acc.c[k / 3][k % 3];
}

// What one call computes at every site of a tile: val = diag * same(site) + hsgn * (-kappa H in)(site).
struct FixOp {
    int dag;             // the hopping term of D^dag
    int parity;          // -1: every site; 0 / 1: the sites of that parity (tile index = half index)
    FixView in;          // full fields, or half vectors of the other parity
    int diag;            // 1: same is added
    int hsgn;            // +1 or -1
    FixView same;
};

// sums of the eight directions for one complex component: SPIN 0 (upper, component c = 3 spin + colour of
// r) and the two lower spins, rebuilt from r by the projectors (signs for D; the caller flips the lower
// ones for D^dag).  R: [8][12][32] (re, im interleaved: component 2c + part), D: alignment shifts.
template <int SPIN>
__device__ __forceinline__ void fix_gather(const long long* R, const int (&D)[8], int c, int lane, long long& re,
                                           long long& im) {
    re = 0;
    im = 0;
#pragma unroll
    for (int d = 0; d < 8; d++) {
        const int mu = d >> 1, back = d & 1;
        // r component (0 or 1) and factor of the rebuilt spin: +-1 or +-i times S, S = -1 forward, +1 backward in D
        int comp = 0, isi = 0, pos = 1;
        if (SPIN == 2) {
            comp = (mu < 2) ? 1 : 0;
            isi = (mu == 0 || mu == 2);
        } else if (SPIN == 3) {
            comp = (mu < 2) ? 0 : 1;
            isi = (mu == 0 || mu == 2);
            pos = (mu == 0 || mu == 3);
        }
        const int cc = SPIN == 0 ? c : 3 * comp + c;
        const long long* p = R + ((size_t)d * 12 + 2 * cc) * 32 + lane;
        const long long x = fix_sra(p[0], D[d]), y = fix_sra(p[32], D[d]);
        if (SPIN == 0) {
            re += x;
            im += y;
        } else {
            const bool plus = (back != 0) == (pos != 0);
            if (isi) {   // i (x + i y) = -y + i x
                if (plus) { re -= y; im += x; } else { re += y; im -= x; }
            } else {
                if (plus) { re += x; im += y; } else { re -= x; im -= y; }
            }
        }
    }
}

// One tile of 32 sites, right-hand sides r0, r0 + rstep, ... < nr.  Every thread of the block (256) calls
// it.  epi(r, plane, idx, live, a, b) receives the two finished entries of pair-plane `plane` at tile
// index idx and returns this thread's share of a sum; with Epi::kShare, epi.put(r, tile, total) follows (one thread).
template <class Epi>
__device__ __forceinline__ void fix_tile(const FixDev& F, const FixOp& op, int tile, int r0, int nr, int rstep,
                                         unsigned char* smem, Epi& epi) {
    const Geom& g = F.g;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int nsite = op.parity < 0 ? g.vol : g.vol / 2;
    int idx = tile * 32 + lane;
    const bool live = idx < nsite;
    if (!live) idx = nsite - 1;
    const int s = op.parity < 0 ? idx : eo_site(g, idx, op.parity);
    double* s_share = reinterpret_cast<double*>(smem + 2 * kFixBufBytes);   // [2][8]
    // ---- this warp's direction ----
    const int mu = warp >> 1, back = warp & 1;
    int nsite_idx;   // the neighbour in this direction
    {
        const int str = mu == 0 ? g.stride[0] : mu == 1 ? g.stride[1] : mu == 2 ? g.stride[2] : g.stride[3];
        const int ext = mu == 0 ? g.L[0] : mu == 1 ? g.L[1] : mu == 2 ? g.L[2] : g.L[3];
        const int c = (s / str) % ext;
        nsite_idx = back ? (c == 0 ? s + (ext - 1) * str : s - str) : (c == ext - 1 ? s - (ext - 1) * str : s + str);
    }
    const int vol = g.vol;
    int4 L[9];   // (re hi, re lo, im hi, im lo), transposed and conjugated for a backward hop
    {
        const int4* lp = F.L + (size_t)(mu * 9) * vol + (back ? nsite_idx : s);
#pragma unroll
        for (int a = 0; a < 3; a++)
#pragma unroll
            for (int b = 0; b < 3; b++) {
                int4 z = __ldg(lp + (size_t)(back ? 3 * b + a : 3 * a + b) * vol);
                if (back) {
                    z.z = -z.z;
                    z.w = -z.w;
                }
                L[3 * a + b] = z;
            }
    }
    // projection h0 = p0 + f0 p_q0, h1 = p1 + f1 p_q1 with f = +-1 or +-i (P = 1 + S g_mu)
    const int S = (back ? 1 : -1) * (op.dag ? -1 : 1);
    const bool swap = mu == 0 || mu == 2;
    const int q0 = mu < 2 ? 3 : 2, q1 = 5 - q0;
    const int f0 = mu == 3 ? S : -S, f1 = mu == 0 ? -S : S;
    const unsigned kNeg = 0x80000000u;
    // factor c (times i when swap): re part flips, im part flips
    const unsigned fr0 = swap ? (f0 > 0 ? kNeg : 0u) : (f0 < 0 ? kNeg : 0u), fi0 = f0 < 0 ? kNeg : 0u;
    const unsigned fr1 = swap ? (f1 > 0 ? kNeg : 0u) : (f1 < 0 ? kNeg : 0u), fi1 = f1 < 0 ? kNeg : 0u;
    const double2* pin = op.in.p + (size_t)(nsite_idx >> op.in.half) * op.in.site;
    int buf = 0, rprev = -1;
    for (int r = r0; r < nr; r += rstep, buf ^= 1) {
        long long* R = reinterpret_cast<long long*>(smem + buf * kFixBufBytes);
        int* sE = reinterpret_cast<int*>(smem + buf * kFixBufBytes + 8 * 12 * 32 * sizeof(long long));
        {
            double2 p[12];   // 0-5: spins 0 and 1; 6-8: spin q0; 9-11: spin q1
            const double2* q = pin + (size_t)r * op.in.field;
            auto at = [&](int k) { return q[(size_t)(k >> 1) * op.in.pair + (k & 1)]; };
#pragma unroll
            for (int c = 0; c < 6; c++) p[c] = at(c);
#pragma unroll
            for (int c = 0; c < 3; c++) {
                p[6 + c] = at(3 * q0 + c);
                p[9 + c] = at(3 * q1 + c);
            }
            int ebits[2];   // each half spinor's own exponent: a spin far below the others keeps its digits
#pragma unroll
            for (int v = 0; v < 2; v++) {
                int mx = 0;
#pragma unroll
                for (int c = 3 * v; c < 3 * v + 3; c++) {
                    mx = max(mx, max(__double2hiint(p[c].x) & 0x7fffffff, __double2hiint(p[c].y) & 0x7fffffff));
                    mx = max(mx, max(__double2hiint(p[6 + c].x) & 0x7fffffff, __double2hiint(p[6 + c].y) & 0x7fffffff));
                }
                int E = mx >> 20;
                if (mx != 0 && (E < kFixEMin || E > kFixEMax)) E = kFixBad;
                sE[(v * 8 + warp) * 32 + lane] = E;
                // all zero (E = 0) still needs an exponent that shifts the components out
                ebits[v] = (E == kFixBad || E == 0 ? kFixEMax : E) << 20;
            }
            int hh[6][2], hl[6][2], nh[6], nl[6];   // limbs of h (re, im) and of -im
#pragma unroll
            for (int c = 0; c < 6; c++) {
                const double2 w = p[6 + c];
                const double wr = swap ? w.y : w.x, wi = swap ? w.x : w.y;
                const int eb = ebits[c / 3];
                int a, b, x, y;
                fix_limbs(p[c].x, eb, 0u, a, b);
                fix_limbs(wr, eb, c < 3 ? fr0 : fr1, x, y);
                hh[c][0] = a + x;
                hl[c][0] = b + y;
                fix_limbs(p[c].y, eb, 0u, a, b);
                fix_limbs(wi, eb, c < 3 ? fi0 : fi1, x, y);
                hh[c][1] = a + x;
                hl[c][1] = b + y;
                nh[c] = -hh[c][1];
                nl[c] = -hl[c][1];
            }
#pragma unroll
            for (int a = 0; a < 3; a++)
#pragma unroll
                for (int v = 0; v < 2; v++) {
                    long long Ar = 0, Br = 0, Ai = 0, Bi = 0;
#pragma unroll
                    for (int b = 0; b < 3; b++) {
                        const int4 l = L[3 * a + b];
                        const int c = 3 * v + b;
                        Ar += (long long)l.x * hh[c][0];
                        Br += (long long)l.x * hl[c][0];
                        Br += (long long)l.y * hh[c][0];
                        Ar += (long long)l.z * nh[c];
                        Br += (long long)l.z * nl[c];
                        Br += (long long)l.w * nh[c];
                        Ai += (long long)l.x * hh[c][1];
                        Bi += (long long)l.x * hl[c][1];
                        Bi += (long long)l.y * hh[c][1];
                        Ai += (long long)l.z * hh[c][0];
                        Bi += (long long)l.z * hl[c][0];
                        Bi += (long long)l.w * hh[c][0];
                    }
                    long long* o = R + ((size_t)warp * 12 + 2 * (3 * v + a)) * 32 + lane;
                    o[0] = Ar + (Br >> 27);
                    o[32] = Ai + (Bi >> 27);
                }
        }
        __syncthreads();
        if (Epi::kShare && rprev >= 0 && threadIdx.x == 6 * 32) {
            const double* sh = s_share + (buf ^ 1) * 8;
            epi.put(rprev, tile, ((sh[0] + sh[1]) + (sh[2] + sh[3])) + (sh[4] + sh[5]));
        }
        rprev = r;
        if (warp < 6) {
            // exponents of the half spinors that an output spin takes from the x, y and the z, t directions, the largest of
            // them, and the others' distance from it
            auto shifts = [&](int spin, int (&D)[8]) {
                const int* xy = sE + (spin == 1 || spin == 2 ? 8 * 32 : 0) + lane;
                const int* zt = sE + (spin & 1 ? 8 * 32 : 0) + lane;
                int Em = 0;
#pragma unroll
                for (int d = 0; d < 8; d++) {
                    D[d] = (d < 4 ? xy : zt)[d * 32];
                    Em = max(Em, D[d]);
                }
#pragma unroll
                for (int d = 0; d < 8; d++) D[d] = Em - D[d];
                return Em;
            };
            // the plane's two entries are of one spin, or (warps 1 and 4) of two
            const int spin0 = 2 * warp / 3, spin1 = (2 * warp + 1) / 3;
            int D[8];
            const int E0 = shifts(spin0, D);
            int E1 = E0;
            double2 pa = make_double2(0.0, 0.0), pb = pa;
            if (op.diag) {
                const int si = op.same.half ? idx : s;
                const double2* q = op.same.p + (size_t)r * op.same.field + (size_t)si * op.same.site + (size_t)warp * op.same.pair;
                pa = q[0];
                pb = q[1];
            }
            double2 va, vb;
            // a diagonal entry outside the fixed point's range (and a sum that is not zero) goes the slow way too
            auto far = [&](double x) {
                const int h = __double2hiint(x) & 0x7fffffff;
                return h != 0 && ((h >> 20) < kFixEMin || (h >> 20) > kFixEMax);
            };
            bool slow = E0 == kFixBad || (op.diag && (far(pa.x) || far(pa.y) || far(pb.x) || far(pb.y)));
            long long x0 = 0, y0 = 0, x1 = 0, y1 = 0;
            if (!slow) {
                if (warp < 3) fix_gather<0>(R, D, 2 * warp, lane, x0, y0);
                else if (warp == 3) fix_gather<2>(R, D, 0, lane, x0, y0);
                else if (warp == 4) fix_gather<2>(R, D, 2, lane, x0, y0);
                else fix_gather<3>(R, D, 1, lane, x0, y0);
                if (spin1 != spin0) E1 = shifts(spin1, D);
                if (warp < 3) fix_gather<0>(R, D, 2 * warp + 1, lane, x1, y1);
                else if (warp == 3) fix_gather<2>(R, D, 1, lane, x1, y1);
                else if (warp == 4) fix_gather<3>(R, D, 0, lane, x1, y1);
                else fix_gather<3>(R, D, 2, lane, x1, y1);
                slow = E1 == kFixBad;
            }
            if (slow) {
                double2 c[12];
                fix_chain(F, op.dag, s, op.in, r, c);
                va = c[2 * warp];
                vb = c[2 * warp + 1];
                const double hs = (double)op.hsgn;
                va = make_double2(pa.x + hs * va.x, pa.y + hs * va.y);
                vb = make_double2(pb.x + hs * vb.x, pb.y + hs * vb.y);
            } else {
                const bool neg = (op.hsgn < 0) != (op.dag && warp >= 3);
                if (neg) {
                    x0 = -x0;
                    y0 = -y0;
                    x1 = -x1;
                    y1 = -y1;
                }
                const int H0 = E0 + kFixUnit - F.k, H1 = E1 + kFixUnit - F.k;
                va.x = fix_combine(x0, H0, op.diag, pa.x);
                va.y = fix_combine(y0, H0, op.diag, pa.y);
                vb.x = fix_combine(x1, H1, op.diag, pb.x);
                vb.y = fix_combine(y1, H1, op.diag, pb.y);
            }
            const double part = epi(r, warp, idx, s, live, va, vb);
            if (Epi::kShare) {
                const double t = warp_sum(part);
                if (lane == 0) s_share[buf * 8 + warp] = t;
            }
        }
    }
    if (Epi::kShare && rprev >= 0) {
        __syncthreads();
        if (threadIdx.x == 6 * 32) {
            const double* sh = s_share + (buf ^ 1) * 8;
            epi.put(rprev, tile, ((sh[0] + sh[1]) + (sh[2] + sh[3])) + (sh[4] + sh[5]));
        }
    }
}

// The same for links out of the fixed point's range: block `block` of the `nblocks` that share ntiles tiles and nr fields.
// A warp takes a tile of one field at a time and no barrier, so the chain is formed once per site and bounded by the
// FP64 pipe; with few fields the first blocks do all of it, eight warps each.  Every thread of the block calls it.
// D on 12 fields of 16^3 x 32: 14.6 ms when the gathering warps each formed the chain, 2.5 ms here.
template <class Epi>
__device__ __forceinline__ void fix_plain(const FixDev& F, const FixOp& op, int block, int nblocks, int ntiles, int nr,
                                          Epi& epi) {
    const Geom& g = F.g;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int nsite = op.parity < 0 ? g.vol : g.vol / 2;
    __syncthreads();   // what the block has put into shared memory for the epilogue
    for (long p = block * 8L + warp; p < (long)ntiles * nr; p += nblocks * 8L) {
        const int tile = (int)(p % ntiles), r = (int)(p / ntiles);
        int idx = tile * 32 + lane;
        const bool live = idx < nsite;
        if (!live) idx = nsite - 1;
        const int s = op.parity < 0 ? idx : eo_site(g, idx, op.parity);
        double2 c[12];
        fix_chain(F, op.dag, s, op.in, r, c);
        const double hs = (double)op.hsgn;
        const double2* q = op.same.p + (size_t)r * op.same.field + (size_t)(op.same.half ? idx : s) * op.same.site;
        double part = 0.0;
#pragma unroll 1
        for (int plane = 0; plane < 6; plane++) {
            double2 v[2];
#pragma unroll
            for (int k = 0; k < 2; k++) {
                const double2 z = c[2 * plane + k];
                const double2 d = op.diag ? q[(size_t)plane * op.same.pair + k] : make_double2(0.0, 0.0);
                v[k] = make_double2(d.x + hs * z.x, d.y + hs * z.y);
            }
            part += epi(r, plane, idx, s, live, v[0], v[1]);
        }
        if (Epi::kShare) {
            const double t = warp_sum(part);
            if (lane == 0) epi.put(r, tile, t);
        }
    }
}

// right-hand sides side by side: as many grid rows as keep about eight blocks per SM, so that
// small lattices fill the chip and large ones keep a link in registers for all of them
inline int fix_grid_y(int tiles, int n) {
    const int want = (8 * 152 + tiles - 1) / tiles;
    return want < 1 ? 1 : want < n ? want : n;
}

}  // namespace seedcg
