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

constexpr int kPairPts = 306;     // points of a tile with its ring of one site: 34 x 9, or as many of another shape
constexpr int kPairTX = 32;       // columns of a tile in domains of such a width
constexpr int kPairPerSM = 2;
constexpr int kPairSlots = kPairPerSM * 152;  // blocks of a wave
constexpr int kPairMaxChunks = 64;

struct PairGrid {
    int tx, ty, cols, rows, zc, chunks;  // tiles in x and y, their columns and rows, layers per chunk, chunks
};
NH_HD int pair_blocks(const PairGrid& p) { return p.tx * p.ty * p.chunks; }
NH_HD constexpr int pair_points(int cols, int rows) { return (cols + 2) * (rows + 2); }
NH_HD constexpr int pair_threads(int points) { return (points + 31) / 32 * 32; }

// Place (1 ... cols, 1 ... rows inside the tile, 0 and cols + 1, rows + 1 on its
// ring) of a thread's point: own points first, then two rows, then two columns.
NH_HD void pair_place(int thread, int cols, int rows, int* hx, int* hy)
{
    const int e = thread - cols * rows, hw = cols + 2;
    if (e < 0) {
        *hx = 1 + thread % cols;
        *hy = 1 + thread / cols;
    } else if (e < 2 * hw) {
        *hy = e < hw ? 0 : rows + 1;
        *hx = e < hw ? e : e - hw;
    } else {
        const int j = e - 2 * hw;
        *hy = 1 + (j >> 1) < rows ? 1 + (j >> 1) : rows;
        *hx = (j & 1) ? cols + 1 : 0;
    }
}

struct PairDomain {
    int nx, ny, nz;
};

inline int pair_max_rows(int cols) { return kPairPts / (cols + 2) - 2; }

inline PairGrid pair_split(const PairDomain& d, int cols, int rows, int layers)
{
    const int zc = std::min(layers, d.nz);
    return PairGrid{(d.nx + cols - 1) / cols, (d.ny + rows - 1) / rows, cols, rows, zc, (d.nz + zc - 1) / zc};
}

// Columns of a tile: 32, or a share of the width of 24 to 64 columns (all of a
// narrower domain) where that leaves at least a tenth fewer points a layer.  (The
// kernel then knows its strides only at run time; tiles of 11 to 16 columns read so
// many more sectors than they need that they were slower than tiles of 32:
// 1024x512x8 221 us a pair of steps instead of 159.)  Two steps, tiles of 32 columns |
// these | single steps, us: 9x330x260 93 | 32 | 38, 33x1000x100 214 | 126 | 160,
// 33x38x600 56 | 34 | 36, 48x640x128 181 | 142 | 189, 65x200x64 51 | 39 | 41; of
// 131x97x60 in tiles of 11 columns | 27 | single steps 43 | 36 | 38.
inline int pair_columns(const PairDomain& d)
{
    auto points = [&](int cols) {
        const int rows = pair_max_rows(cols);
        return (double)((d.nx + cols - 1) / cols) * ((d.ny + rows - 1) / rows) * pair_points(cols, rows);
    };
    int best = kPairTX;
    for (int t = 1; t <= d.nx; ++t) {
        const int cols = (d.nx + t - 1) / t;
        if (cols > 64) continue;
        if (cols < 24 && t > 1) break;
        if (points(cols) < (best == kPairTX ? 0.9 : 1.0) * points(best)) best = cols;
    }
    return best;
}

// Rows of a tile and layers per chunk: the blocks run in waves of two per SM, and
// a block takes (layers + 2) x (points of a layer); the split with the least sum
// (256x256x64: 296 blocks of 7 rows and 64 layers).  The channels of a launch share
// the layers and fill the waves together.  A pair of steps of eight channels of
// 128x128x48: 250 us in two waves of whole columns, 277 us with the split that each
// takes alone; of 64x64x200: 270 us, whole columns 495 us; two of 151x117x45: 79 us,
// in chunks of 15 layers 89 us.
inline void pair_plan(const PairDomain* d, int count, PairGrid* out)
{
    int most = 1, less = 0, layers = 1;
    for (int k = 0; k < count; ++k) most = std::max(most, d[k].nz);
    long long cost = -1;
    for (int l = 0; l <= 3; ++l) {
        for (int k = 0; k < count; ++k) {
            const int cols = pair_columns(d[k]);
            out[k] = pair_split(d[k], cols, std::max(1, pair_max_rows(cols) - l), d[k].nz);
        }
        for (int n = 1; n <= most && n <= kPairMaxChunks; ++n) {
            const int zc = (most + n - 1) / n;
            long long blocks = 0;
            int points = 0;
            for (int k = 0; k < count; ++k) {
                blocks += (long long)out[k].tx * out[k].ty * ((d[k].nz + zc - 1) / zc);
                points = std::max(points, pair_points(out[k].cols, out[k].rows));
            }
            const long long w = (blocks + kPairSlots - 1) / kPairSlots * (zc + 2) * points;
            if (cost < 0 || w < cost) {
                cost = w;
                less = l;
                layers = zc;
            }
        }
    }
    for (int k = 0; k < count; ++k) {
        const int cols = pair_columns(d[k]);
        out[k] = pair_split(d[k], cols, std::max(1, pair_max_rows(cols) - less), layers);
    }
}

// The kernel's 32-bit byte offsets within the populations.
inline bool pair_offsets_fit(const PairDomain& d) { return 19.0 * 4.0 * d.nx * d.ny * d.nz < 4294967296.0; }
// No more blocks than the diagnostics' partials (of single channels) have room for.
inline bool pair_partials_fit(const PairDomain& d, const PairGrid& p)
{
    return pair_blocks(p) <= ((double)d.nx * d.ny * d.nz + 127) / 128;
}

// From 7.5e5 sites, where the two population buffers no longer stay in L2 (16 LB
// steps and an FD update, single steps | pairs, us: 128x128x32 191 | 212,
// 160x128x32 271 | 279, 128x128x48 329 | 315, 256x256x12 335 | 306, 180x140x32 353 |
// 343, 151x117x45 394 | 335, 256x256x64 1798 | 1388), and up to 2.5 points of the
// first step a site, rings and the layers at the ends of a march included
// (256x256x64: 1.4; two steps, single | pair, us: 1024x512x3, 2.3 points, 78 | 70,
// 1024x1024x2, 2.75 points, 102 | 104, 2048x2048x1, 4.1 points, 201 | 242).
constexpr double kPairMinSites = 7.5e5, kPairMaxPoints = 2.5;
inline bool pair_pays(const PairDomain& d, const PairGrid& p)
{
    const double N = (double)d.nx * d.ny * d.nz;
    return N >= kPairMinSites && (double)pair_blocks(p) * (p.zc + 2) * pair_points(p.cols, p.rows) <= kPairMaxPoints * N;
}

}  // namespace nh
