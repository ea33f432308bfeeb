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
    std::printf("%s: %d x %d x %d, %d x %d tiles of %d rows, %d chunks of %d\n", what, d.nx, d.ny, d.nz, p.tx, p.ty, p.rows,
                p.chunks, p.zc);
}
static bool covers(int tiles, int size, int n) { return tiles * size >= n && (tiles - 1) * size < n; }

// waves of blocks x points of a block, the measure of a launch
static long long cost(const PairGrid* p, size_t n)
{
    long long blocks = 0, zc = 0;
    for (size_t k = 0; k < n; ++k) {
        blocks += pair_blocks(p[k]);
        zc = std::max<long long>(zc, p[k].zc);
    }
    return (blocks + kPairSlots - 1) / kPairSlots * (zc + 2) * (p[0].rows + 2);
}

static void check(const std::vector<PairDomain>& d)
{
    std::vector<PairGrid> p(d.size()), q(d.size());
    pair_plan(d.data(), (int)d.size(), p.data());
    int most = 1;
    for (size_t k = 0; k < d.size(); ++k) {
        want(covers(p[k].tx, kPairTX, d[k].nx) && covers(p[k].ty, p[k].rows, d[k].ny) && covers(p[k].chunks, p[k].zc, d[k].nz),
             "tiles and chunks cover the channel once", d[k], p[k]);
        want(p[k].rows >= 1 && p[k].rows <= kPairTY && p[k].rows == p[0].rows, "rows that all channels share", d[k], p[k]);
        want(kPairHX * (p[k].rows + 2) <= kPairPts && pair_threads(p[k].rows) <= pair_threads(kPairTY), "points of a block", d[k], p[k]);
        most = std::max(most, d[k].nz);
    }
    for (int rows = 4; rows <= kPairTY; ++rows)
        for (int n = 1; n <= most && n <= kPairMaxChunks; ++n) {
            for (size_t k = 0; k < d.size(); ++k) q[k] = pair_split(d[k], rows, (most + n - 1) / n);
            want(cost(p.data(), p.size()) <= cost(q.data(), q.size()), "no better split", d[0], q[0]);
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
    check({{1, 1, 1}});
    check({{2000, 6, 64}, {9, 330, 260}, {1024, 750, 1}});
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
