"""Bookkeeping of the kernels' opt-in to large dynamic shared memory
(csrc/shs_device_once.h): once per device, again after a failure, from several
threads; and no launcher keeps the opt-in per process."""

import glob
import os
import re
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2104_00359_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <thread>
#include <vector>
#include "shs_device_once.h"

#define CHECK(c) do { if (!(c)) { std::printf("line %d: %s\n", __LINE__, #c); return 1; } } while (0)

int main() {
    std::atomic<int> set[80]{};   // opt-ins made per device
    shs::DeviceOnce once;
    auto call = [&](int dev, int status) { return once.run(dev, [&] { ++set[dev]; return status; }); };
    CHECK(call(0, 0) == 0 && call(0, 0) == 0 && set[0] == 1);
    CHECK(call(1, 0) == 0 && set[1] == 1);                       // the second device has its own
    CHECK(call(63, 0) == 0 && call(63, 0) == 0 && set[63] == 1);
    CHECK(call(2, 7) == 7 && call(2, 0) == 0 && call(2, 0) == 0 && set[2] == 2);
    CHECK(call(64, 0) == 0 && call(64, 0) == 0 && set[64] == 2);   // past the bookkeeping: every time
    CHECK(call(79, 3) == 3 && set[79] == 1 && set[15] == 0 && call(15, 0) == 0 && set[15] == 1);
    std::vector<std::thread> threads;
    std::atomic<int> bad{0};
    for (int t = 0; t < 8; ++t)
        threads.emplace_back([&] { for (int dev = 16; dev < 48; ++dev) bad += call(dev, 0) != 0; });
    for (auto& t : threads) t.join();
    for (int dev = 16; dev < 48; ++dev) {
        const int before = set[dev];
        CHECK(before >= 1 && call(dev, 0) == 0 && set[dev] == before);
    }
    CHECK(bad == 0);
    return 0;
}
"""


def test_once_per_device(tmp_path):
    src, exe = tmp_path / "once.cpp", tmp_path / "once"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-O2", "-pthread", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout


def test_no_opt_in_per_process():
    for path in glob.glob(os.path.join(CSRC, "*.cu*")) + glob.glob(os.path.join(CSRC, "*.h")):
        text = open(path).read()
        assert not re.search(r"static\s+(const\s+)?cudaError_t[^;(]*=[^;]*cudaFuncSetAttribute", text), path
