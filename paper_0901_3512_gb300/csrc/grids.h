// Launch grids of the Lanczos kernels and the size of the reduction workspace that they share.  Host code only
// (no CUDA), so that the sizes can be checked without a GPU.
#pragma once

#include <algorithm>
#include <cstddef>

namespace seedcg {

constexpr int kRedThreads = 256;  // every reducing kernel uses this block size
constexpr int kMaxRedBlocks = 4096;

inline int red_blocks(long n) {
    long b = (n + kRedThreads * 4 - 1) / (kRedThreads * 4);
    if (b < 1) b = 1;
    return (int)std::min<long>(b, 152 * 8);
}

// blocks for a kernel whose thread handles one 16-byte group of entries (n / w
// groups), in equal rounds of at most kMaxRedBlocks blocks
inline int vec_blocks(long n, int w) {
    long b = (n / w + kRedThreads - 1) / kRedThreads;
    if (b < 1) b = 1;
    const long rounds = (b + kMaxRedBlocks - 1) / kMaxRedBlocks;
    return (int)((b + rounds - 1) / rounds);
}

inline int site_blocks(int vol) { return (vol + kRedThreads - 1) / kRedThreads; }

// The single-RHS operator kernels of the Lanczos loop (one thread per site) run in
// blocks of 128 with at most 72 registers in FP32: 7 blocks per SM then hold a
// 16^3x32 lattice in one wave, where 256-thread blocks at 77 registers need 1.12
// waves (16.4 -> 14.6 us for D with the L2 warm)
constexpr int kSiteThreads = 128;
inline int site_blocks_lz(int vol) { return (vol + kSiteThreads - 1) / kSiteThreads; }

inline int fix_tiles(int sites) { return (sites + 31) / 32; }              // the FP64 operator: 32 sites per block
inline long entry_blocks(long n, int w) { return (n / w + kRedThreads - 1) / kRedThreads; }   // w entries per thread

// Doubles that the kernels of one Lanczos run may write as block partials (grid_sum: NV per block) on vectors of
// n = 12 * sites entries: the operator's last kernel (one thread per site, or one block per 32 sites in FP64), the
// literal seeds (16 per block), the FP64 subtraction of a re-orthogonalisation (one entry per thread) and the
// streaming passes.  The first term has been the size of this workspace for every lattice up to about 5 million sites.
inline size_t lz_partial_doubles(long n, int nrhs, bool fp64) {
    const int sites = (int)(n / 12), rb = red_blocks(n);
    size_t d = (size_t)std::max(kMaxRedBlocks, rb * (nrhs + 2)) * 64;
    d = std::max(d, (size_t)(fp64 ? fix_tiles(sites) : site_blocks_lz(sites)));
    if (fp64) d = std::max(d, (size_t)entry_blocks(n, 1));
    return std::max(d, (size_t)16 * rb);
}

}  // namespace seedcg
