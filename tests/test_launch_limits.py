"""The shared-memory limit of a kernel (csrc/launch_limits.cuh), compiled for the
host with a slow setter: threads that ask for different sizes at once never leave
it below what any of them was told it may launch with."""

import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2304_14492_gb300", "csrc")

PROGRAM = r'''
#include <chrono>
#include <cstdio>
#include <thread>
#include <vector>
#include "launch_limits.cuh"

int main() {
    using std::chrono::microseconds;
    for (int dev : {0, 3, 63, 64, 70})
        for (int round = 0; round < 20; ++round) {
            zm::SharedMemoryLimit limit;
            std::atomic<size_t> attribute{48 << 10};
            std::atomic<int> sets{0}, bad{0};
            auto ask = [&](size_t bytes) {
                const int e = limit.raise(dev, bytes, [&](size_t n) {
                    std::this_thread::sleep_for(microseconds(300 - n / 1024));   // smaller sizes arrive later
                    attribute = n;
                    ++sets;
                    return 0;
                });
                for (int k = 0; k < 20; ++k) {                                   // from now on it may launch
                    if (e != 0 || attribute < bytes) ++bad;
                    std::this_thread::sleep_for(microseconds(50));
                }
            };
            std::vector<std::thread> ts;
            for (int t = 0; t < 12; ++t) ts.emplace_back(ask, (size_t)(8 + 18 * ((t * 7 + round) % 12)) << 10);
            for (auto& t : ts) t.join();
            if (bad || attribute != (size_t)(8 + 18 * 11) << 10 || sets > 12) return 1;
            // an error is passed on and leaves the limit where it was
            if (limit.raise(dev, 227 << 10, [](size_t) { return 7; }) != 7) return 2;
            int again = 0;
            if (limit.raise(dev, 227 << 10, [&](size_t) { return ++again, 0; }) != 0 || again != 1) return 3;
            if (limit.raise(dev, 100 << 10, [&](size_t) { return 9; }) != 0) return 4;
            if (limit.raise(dev + 1, 60 << 10, [&](size_t) { return ++again, 0; }) != 0 || again != 2) return 5;
        }
    return 0;
}
'''


def test_threads_never_lower_it(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no host compiler")
    (tmp_path / "t.cpp").write_text(PROGRAM)
    exe = str(tmp_path / "t")
    subprocess.run([cxx, "-O2", "-std=c++17", "-pthread", "-I" + CSRC, str(tmp_path / "t.cpp"), "-o", exe], check=True)
    assert subprocess.run([exe], timeout=120).returncode == 0
