// pair_plan.h -- how the kernel that takes two LB steps in one pass (lb.cu) cuts channels into tiles and marches.
// Plain C++: the host plans with it, the kernel reads the result.
#pragma once

#include <algorithm>

#ifdef __CUDACC__
#define NH_HD __host__ __device__ __forceinline__
#else
#define NH_HD inline
#endif

namespace nh {

constexpr int kPairTX = 32, kPairTY = 7;  // columns and, at most, rows of a tile
constexpr int kPairHX = kPairTX + 2, kPairHY = kPairTY + 2, kPairPts = kPairHX * kPairHY;  // with its ring
constexpr int kPairPerSM = 2;
constexpr int kPairSlots = kPairPerSM * 152;  // blocks of a wave
constexpr int kPairMaxChunks = 64;

struct PairGrid {
    int tx, ty, rows, zc, chunks;  // tiles in x and y, rows of a tile, layers per chunk, chunks
};
NH_HD int pair_blocks(const PairGrid& p) { return p.tx * p.ty * p.chunks; }
NH_HD constexpr int pair_threads(int rows) { return (kPairHX * (rows + 2) + 31) / 32 * 32; }

struct PairDomain {
    int nx, ny, nz;
};

inline PairGrid pair_split(const PairDomain& d, int rows, int layers)
{
    const int zc = std::min(layers, d.nz);
    return PairGrid{(d.nx + kPairTX - 1) / kPairTX, (d.ny + rows - 1) / rows, rows, zc, (d.nz + zc - 1) / zc};
}

// Rows of a tile and layers per chunk: the blocks run in waves of two per SM, and
// a block takes (layers + 2) x (points of a layer); the split with the least sum
// (256x256x64: 296 blocks of 7 rows and 64 layers).  The channels of a launch share
// both numbers and fill the waves together.  A pair of steps of eight channels of
// 128x128x48: 258 us in two waves of whole columns, 277 us with the split that each
// takes alone; of 64x64x200: 282 us, whole columns 495 us; two of 151x117x45: 82 us,
// in chunks of 15 layers 89 us.
inline void pair_plan(const PairDomain* d, int count, PairGrid* out)
{
    int most = 1, rows = kPairTY, layers = 1;
    for (int k = 0; k < count; ++k) most = std::max(most, d[k].nz);
    long long cost = -1;
    for (int r = kPairTY; r >= 4; --r)
        for (int n = 1; n <= most && n <= kPairMaxChunks; ++n) {
            const int zc = (most + n - 1) / n;
            long long blocks = 0;
            for (int k = 0; k < count; ++k) blocks += pair_blocks(pair_split(d[k], r, zc));
            const long long w = (blocks + kPairSlots - 1) / kPairSlots * (zc + 2) * (r + 2);
            if (cost < 0 || w < cost) {
                cost = w;
                rows = r;
                layers = zc;
            }
        }
    for (int k = 0; k < count; ++k) out[k] = pair_split(d[k], rows, layers);
}

// The kernel's 32-bit byte offsets within the populations.
inline bool pair_offsets_fit(const PairDomain& d) { return 19.0 * 4.0 * d.nx * d.ny * d.nz < 4294967296.0; }
// No more blocks than the diagnostics' partials (of single channels) have room for.
inline bool pair_partials_fit(const PairDomain& d, const PairGrid& p)
{
    return pair_blocks(p) <= ((double)d.nx * d.ny * d.nz + 127) / 128;
}

// From 7.5e5 sites, where the two population buffers no longer stay in L2 (16 LB
// steps and an FD update, single steps | pairs, us: 128x128x32 195 | 218,
// 160x128x32 275 | 288, 128x128x48 337 | 323, 256x256x12 343 | 315, 180x140x32 355 |
// 355, 151x117x45 407 | 349, 256x256x64 1815 | 1446).
constexpr double kPairMinSites = 7.5e5;
inline bool pair_pays(const PairDomain& d) { return (double)d.nx * d.ny * d.nz >= kPairMinSites; }

}  // namespace nh
