"""Host state kept per device: what holds on one device is not taken to hold on
another (kernel attributes are set where the kernel runs)."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2510_07672_gb300", "csrc")

MAIN = r"""
#include <cstdio>
#include <thread>
#include <vector>
#include "per_device.cuh"
int main() {
    acpr::DeviceSet s;
    if (s.has(0) || s.has(1)) return 1;
    s.add(0);
    if (!s.has(0) || s.has(1) || s.has(63)) return 2;
    s.add(64);   // beyond the set: never remembered, so set again on each call
    s.add(-1);
    if (s.has(64) || s.has(-1) || s.has(1)) return 3;
    std::vector<std::thread> t;
    for (int d = 0; d < 64; ++d) t.emplace_back([&s, d] { s.add(d); });
    for (auto& x : t) x.join();
    for (int d = 0; d < 64; ++d)
        if (!s.has(d)) return 4;
    return 0;
}
"""


def test_device_set(tmp_path):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no host compiler")
    (tmp_path / "main.cc").write_text(MAIN)
    exe = str(tmp_path / "main")
    subprocess.check_call([cxx, "-std=c++17", "-pthread", "-I", CSRC, str(tmp_path / "main.cc"), "-o", exe])
    assert subprocess.run([exe]).returncode == 0


def test_every_kernel_attribute_is_set_per_device():
    """Kernel attributes are set in one place, under a set of devices."""
    for name in sorted(os.listdir(CSRC)):
        text = open(os.path.join(CSRC, name)).read()
        assert ("cudaFuncSetAttribute" in text) == (name == "common.cuh"), name
        assert "static bool configured" not in text, name
