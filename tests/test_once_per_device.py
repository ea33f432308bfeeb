"""Set-up that belongs to a device (the kernels' opt-in to large shared memory)
runs once for every device of a process, whatever thread comes first."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2503_06610_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <thread>
#include <vector>
#include "once_per_device.h"
static int fails = 0;
static void want(bool ok, const char* what) { if (!ok) { std::printf("%s\n", what); fails = 1; } }
int main()
{
    nh::OncePerDevice once;
    int runs[70] = {};
    auto set = [&](int d, int status) { return once(d, [&] { ++runs[d]; return status; }); };
    want(set(0, 0) == 0 && set(0, 0) == 0 && runs[0] == 1, "once on device 0");
    want(set(1, 0) == 0 && runs[1] == 1, "device 1 has its own");
    want(set(0, 0) == 0 && set(1, 0) == 0 && runs[0] == 1 && runs[1] == 1, "neither again");
    want(set(2, 7) == 7 && set(2, 0) == 0 && set(2, 0) == 0 && runs[2] == 2, "a failure is returned and tried again");
    want(set(63, 0) == 0 && set(63, 0) == 0 && runs[63] == 1, "the last device that is remembered");
    want(set(64, 0) == 0 && set(64, 0) == 0 && runs[64] == 2, "beyond it: every time");
    nh::OncePerDevice shared;
    std::atomic<int> calls{0};
    std::vector<std::thread> threads;
    for (int t = 0; t < 8; ++t)
        threads.emplace_back([&] { for (int k = 0; k < 1000; ++k) shared(k % 4, [&] { ++calls; return 0; }); });
    for (auto& t : threads) t.join();
    want(calls >= 4 && calls <= 32, "a few runs from eight threads");
    return fails;
}
"""


def test_once_per_device(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    src, exe = tmp_path / "once.cpp", tmp_path / "once"
    src.write_text(PROGRAM)
    subprocess.run([cxx, "-std=c++17", "-O1", "-pthread", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    res = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert res.returncode == 0, res.stdout


def test_no_opt_in_is_remembered_per_process():
    for name in sorted(os.listdir(CSRC)):
        with open(os.path.join(CSRC, name)) as f:
            assert "static bool" not in f.read(), name + ": a flag of the process stands for every device"
