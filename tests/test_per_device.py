"""What launches keep per device (csrc/per_device.h): made once for each device, never for another, and
not kept when it failed.  Host code, built with the host compiler."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2403_01254_gb300", "csrc")

PROGRAM = r"""
#include "per_device.h"
#include <cstdio>
#include <thread>
#include <vector>
int main() {
    static rk::PerDevice cache;
    int made = 0;
    for (int round = 0; round < 3; ++round)
        for (int dev : {0, 1, 7, 63})
            if (cache.get(dev, [&] { ++made; return 10 + dev; }) != 10 + dev) return 1;
    if (made != 4) return 2;                                  // once for each device
    int tries = 0;
    if (cache.get(2, [&] { ++tries; return 0; }) != 0) return 3;
    if (cache.get(2, [&] { ++tries; return 5; }) != 5) return 4;
    if (cache.get(2, [&] { ++tries; return 6; }) != 5 || tries != 2) return 5;     // a failure is not kept
    for (int dev : {64, 1000, -1})
        for (int v : {3, 4})
            if (cache.get(dev, [&] { return v; }) != v) return 6;                  // asked each time
    static rk::PerDevice shared;
    std::vector<std::thread> ts;
    std::atomic<int> bad{0};
    for (int t = 0; t < 8; ++t)
        ts.emplace_back([&, t] {
            for (int i = 0; i < 20000; ++i)
                if (shared.get(i & 3, [&] { return 1 + (i & 3); }) != 1 + (i & 3)) ++bad;
        });
    for (auto& t : ts) t.join();
    return bad ? 7 : 0;
}
"""


def test_per_device_values(tmp_path):
    gxx = shutil.which("g++")
    if not gxx:
        pytest.skip("no host compiler")
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(PROGRAM)
    subprocess.run([gxx, "-std=c++17", "-O1", "-pthread", "-I" + CSRC, str(src), "-o", str(exe)], check=True)
    assert subprocess.run([str(exe)]).returncode == 0


def test_no_launch_keeps_a_device_property_for_the_process():
    # every opt-in to shared memory beyond 48 KB goes through the cache above
    for f in os.listdir(CSRC):
        if not f.endswith(".cu"):
            continue
        text = open(os.path.join(CSRC, f)).read()
        for word in ("static int resident", "static bool attr_set", "static std::atomic<bool> opted"):
            assert word not in text, (f, word)
