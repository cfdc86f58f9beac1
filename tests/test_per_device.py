"""Values that belong to a device (a function attribute, an occupancy) are found once for each device of the process,
failures are asked for again, and no kernel's attribute is set for the first device alone."""
import glob
import os
import re
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2605_10760_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <thread>
#include <vector>
#include "gs_device.cuh"
int main() {
    gs::PerDevice v;
    int calls[3] = {0, 0, 0};
    for (int r = 0; r < 3; ++r)
        for (int d = 0; d < 3; ++d)
            if (v.get(d, [&] { ++calls[d]; return 10 + d; }) != 10 + d) return 1;
    if (calls[0] != 1 || calls[1] != 1 || calls[2] != 1) return 2;
    gs::PerDevice f;
    int n = 0;
    auto third = [&] { return ++n < 3 ? 0 : 7; };
    if (f.get(0, third) != 0 || f.get(0, third) != 0 || f.get(0, third) != 7 || f.get(0, third) != 7 || n != 3) return 3;
    if (f.get(-1, [] { return 5; }) != 5 || f.get(1000, [] { return 6; }) != 6) return 4;
    gs::PerDevice t;
    std::vector<std::thread> threads;
    for (int k = 0; k < 8; ++k) threads.emplace_back([&] { for (int d = 0; d < 64; ++d) if (t.get(d, [d] { return d + 1; }) != d + 1) std::puts("bad"); });
    for (auto &x : threads) x.join();
    std::puts("ok");
}
"""


def test_one_value_per_device(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no host compiler")
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(PROGRAM)
    subprocess.run([gxx, "-std=c++17", "-pthread", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True)
    assert (r.returncode, r.stdout) == (0, "ok\n")


def test_attributes_are_set_on_every_device():
    for path in glob.glob(os.path.join(CSRC, "*.cu")):
        code = open(path).read()
        for m in re.finditer(r"cudaFuncSetAttribute", code):
            before = code[max(0, m.start() - 120):m.start()]
            assert ".get(" in before and not re.search(r"static \w+ \w+ =\s*$", before), path
