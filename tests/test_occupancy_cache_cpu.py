"""The kept answers of the occupancy queries (csrc/gs_occupancy.h), compiled by the host
compiler: one query per kernel, size and device, in any order and from several
threads; failures and a full table are asked again."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2409_13055_gb300", "csrc")
SOURCE = r"""
#include <atomic>
#include <cstdio>
#include <thread>
#include <vector>
#include "gs_occupancy.h"
#define CHECK(x) do { if (!(x)) { std::printf("line %d: %s\n", __LINE__, #x); return 1; } } while (0)
int main() {
    static gs::OccupancyCache c;
    const char kernels[400] = {};
    std::atomic<int> asked{0};
    auto get = [&](int k, int threads, size_t smem, int dev) {
        return c.get(kernels + k, threads, smem, dev, [&] {
            ++asked;
            return 1 + k + threads + (int)smem + 1000 * dev;
        });
    };
    // the sizes of a plan's depth and tile passes in turn, on two devices
    for (int turn = 0; turn < 5; ++turn)
        for (int dev = 0; dev < 2; ++dev)
            for (size_t smem : {8192u, 4096u, 512u})
                for (int k = 0; k < 3; ++k)
                    CHECK(get(k, 256, smem, dev) == 1 + k + 256 + (int)smem + 1000 * dev);
    CHECK(asked == 18);
    CHECK(get(0, 128, 512, 0) == 1 + 128 + 512 && asked == 19);
    int failed = 0;
    for (int i = 0; i < 2; ++i)
        CHECK(c.get(kernels + 399, 1, 0, 0, [&] { ++failed; return -1; }) == -1);
    CHECK(failed == 2);
    std::vector<std::thread> all;
    for (int t = 0; t < 8; ++t)
        all.emplace_back([&] {
            for (int i = 0; i < 200; ++i) get(10 + i % 20, 256, 64, 0);
        });
    for (auto& t : all) t.join();
    CHECK(asked == 39);
    for (int i = 0; i < 300; ++i) CHECK(get(i, 7, 7, 0) == 15 + i);  // beyond the table
    for (int i = 0; i < 300; ++i) CHECK(get(i, 7, 7, 0) == 15 + i);
    return 0;
}
"""


def test_every_key_is_asked_once(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if not cxx:
        pytest.skip("no host C++ compiler")
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(SOURCE)
    subprocess.run([cxx, "-std=c++17", "-O1", "-pthread", "-I", CSRC, str(src), "-o", str(exe)],
                   check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
