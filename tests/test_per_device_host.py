"""Kernel attributes, SM counts and symbol addresses are made once for every
device of a process, not once for the process (csrc/per_device.h, host code)."""

import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1607_02573_gb300", "csrc")

MAIN = """
#include <cstdio>
#include <stdexcept>
#include <thread>
#include <vector>
#include "per_device.h"

int main() {
    mwi::PerDevice<int> v;
    int made[2] = {0, 0}, failed = 0;
    try {
        v.get(1, []() -> int { throw std::runtime_error("not this time"); });
    } catch (const std::runtime_error&) {
        ++failed;
    }
    std::vector<std::thread> t;
    bool same = true;
    for (int k = 0; k < 8; ++k)
        t.emplace_back([&, k] {
            const int dev = k % 2;
            if (v.get(dev, [&] { ++made[dev]; return 10 + dev; }) != 10 + dev) same = false;
        });
    for (auto& x : t) x.join();
    std::printf("%d %d %d %d", failed, made[0], made[1], same ? 1 : 0);
    return 0;
}
"""


def test_values_are_made_once_for_every_device(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    (tmp_path / "main.cpp").write_text(MAIN)
    exe = str(tmp_path / "main")
    subprocess.run([cxx, "-std=c++17", "-pthread", "-I", CSRC, str(tmp_path / "main.cpp"), "-o", exe], check=True)
    assert subprocess.run([exe], capture_output=True, text=True, check=True).stdout == "1 1 1 1"

