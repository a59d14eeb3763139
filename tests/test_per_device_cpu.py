"""Figures kept per device: each device's own, found once, also from several
threads; and no host function keeps one device's figure for all of them."""
import glob
import os
import re
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2602_14975_gb300", "csrc")

PROBE = r"""
#include <cstdio>
#include <thread>
#include <vector>
#include "per_device.h"
int main() {
    static dmts::PerDevice p;
    std::atomic<int> found{0}, wrong{0};
    std::vector<std::thread> t;
    for (int k = 0; k < 8; ++k)
        t.emplace_back([&, k] {
            for (int i = 0; i < 10000; ++i) {
                const int dev = (i + k) % 70 - 2;   // ordinals outside the table too
                if (p.get(dev, [&] { ++found; return 100 + dev; }) != 100 + dev) ++wrong;
            }
        });
    for (auto &x : t) x.join();
    const int before = found;
    for (int dev = 0; dev < 64; ++dev)
        if (p.get(dev, [&] { ++found; return -1; }) != 100 + dev) ++wrong;
    std::printf("%d %d\n", (int)wrong, (int)found - before);
    return 0;
}
"""


def test_each_device_keeps_its_own_figure(tmp_path):
    src, exe = tmp_path / "probe.cpp", tmp_path / "probe"
    src.write_text(PROBE)
    subprocess.run(["g++", "-std=c++17", "-O1", "-pthread", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    assert subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout.split() == ["0", "0"]


def test_no_host_function_keeps_one_devices_figure():
    for path in glob.glob(os.path.join(CSRC, "*.cu*")):
        assert not re.search(r"^\s+static int \w+ *(=|;)", open(path).read(), re.M), path
