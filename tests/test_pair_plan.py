"""How the kernel that takes two LB steps in one pass cuts channels: host rules,
compiled here without CUDA."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2503_06610_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <random>
#include <vector>
#include "pair_plan.h"
using namespace nh;

static int fails = 0;
static void want(bool ok, const char* what, const PairDomain& d, const PairGrid& p)
{
    if (ok) return;
    fails = 1;
    std::printf("%s: %d x %d x %d, %d x %d tiles of %d x %d, %d chunks of %d\n", what, d.nx, d.ny, d.nz, p.tx, p.ty, p.cols, p.rows,
                p.chunks, p.zc);
}
static bool covers(int tiles, int size, int n) { return tiles * size >= n && (tiles - 1) * size < n; }

// waves of blocks x points of a block, the measure of a launch
static long long cost(const std::vector<PairGrid>& p, int layers)
{
    long long blocks = 0;
    int points = 0;
    for (const PairGrid& g : p) {
        blocks += pair_blocks(g);
        points = std::max(points, pair_points(g.cols, g.rows));
    }
    return (blocks + kPairSlots - 1) / kPairSlots * (layers + 2) * points;
}

// every point of a tile with its ring has one thread, the tile's own points the first
static bool places(int cols, int rows)
{
    std::vector<int> seen((cols + 2) * (rows + 2), 0);
    for (int t = 0; t < pair_points(cols, rows); ++t) {
        int hx, hy;
        pair_place(t, cols, rows, &hx, &hy);
        if (hx < 0 || hx > cols + 1 || hy < 0 || hy > rows + 1) return false;
        ++seen[hx + (cols + 2) * hy];
        const bool inside = hx >= 1 && hx <= cols && hy >= 1 && hy <= rows;
        if (inside != (t < cols * rows)) return false;
    }
    for (int n : seen)
        if (n != 1) return false;
    return true;
}

static void check(const std::vector<PairDomain>& d)
{
    std::vector<PairGrid> p(d.size()), q(d.size());
    pair_plan(d.data(), (int)d.size(), p.data());
    int most = 1, layers = 1;
    for (size_t k = 0; k < d.size(); ++k) {
        want(covers(p[k].tx, p[k].cols, d[k].nx) && covers(p[k].ty, p[k].rows, d[k].ny) && covers(p[k].chunks, p[k].zc, d[k].nz),
             "tiles and chunks cover the channel once", d[k], p[k]);
        want(p[k].cols >= 1 && p[k].rows >= 1 && pair_points(p[k].cols, p[k].rows) <= kPairPts, "points of a block", d[k], p[k]);
        want(places(p[k].cols, p[k].rows), "a thread for every point", d[k], p[k]);
        const PairGrid wide = pair_split(d[k], kPairTX, pair_max_rows(kPairTX), p[k].zc);
        if (p[k].rows == pair_max_rows(p[k].cols))
            want((double)p[k].tx * p[k].ty * pair_points(p[k].cols, p[k].rows) <=
                     (double)wide.tx * wide.ty * pair_points(wide.cols, wide.rows),
                 "no more points than tiles of 32 columns", d[k], p[k]);
        most = std::max(most, d[k].nz);
        layers = std::max(layers, p[k].zc);
    }
    for (int less = 0; less <= 3; ++less)
        for (int n = 1; n <= most && n <= kPairMaxChunks; ++n) {
            const int zc = (most + n - 1) / n;
            for (size_t k = 0; k < d.size(); ++k) {
                const int cols = pair_columns(d[k]);
                q[k] = pair_split(d[k], cols, std::max(1, pair_max_rows(cols) - less), zc);
            }
            want(cost(p, layers) <= cost(q, zc), "no better split", d[0], q[0]);
        }
}

int main()
{
    std::mt19937 rng(5);
    auto upto = [&](int n) { return 1 + (int)(rng() % n); };
    for (int k = 0; k < 400; ++k) {
        std::vector<PairDomain> d(k % 2 ? 1 : upto(12));
        for (auto& g : d) g = PairDomain{upto(300), upto(300), upto(k % 3 ? 90 : 400)};
        check(d);
    }
    for (int nx = 1; nx <= 130; ++nx) check({{nx, 1000 / nx + 1, 40}});
    check({{1, 1, 1}});
    check({{2000, 6, 64}, {9, 330, 260}, {1024, 750, 1}});
    // narrow and wide domains take pairs, domains of a layer or two do not
    const PairDomain pays[] = {{256, 256, 64}, {33, 1000, 23}, {33, 38, 600}, {9, 330, 260}, {65, 200, 64}, {1024, 1024, 4}};
    const PairDomain not_[] = {{1024, 750, 1}, {768, 512, 2}, {96, 96, 32}, {1, 1000, 800}};
    for (const PairDomain& d : pays) {
        PairGrid p;
        pair_plan(&d, 1, &p);
        want(pair_pays(d, p) && pair_partials_fit(d, p), "takes pairs", d, p);
    }
    for (const PairDomain& d : not_) {
        PairGrid p;
        pair_plan(&d, 1, &p);
        want(!pair_pays(d, p), "takes single steps", d, p);
    }
    return fails;
}
"""


def test_pair_plan(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    src, exe = tmp_path / "plan.cpp", tmp_path / "plan"
    src.write_text(PROGRAM)
    subprocess.run([cxx, "-std=c++17", "-O1", "-Wall", "-Werror", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    res = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    assert res.returncode == 0, res.stdout
