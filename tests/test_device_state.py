"""What belongs to a device is set up on each device, not once in the process:
kernels' function attributes and what is asked about their launches.  CPU checks
of the table that prep_conv keeps and of the sources."""
import os
import re
import shutil
import subprocess

import pytest

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1901_08269_gb300", "csrc")


def test_no_attribute_is_set_by_a_static_initialiser():
    for f in sorted(os.listdir(SRC)):
        with open(os.path.join(SRC, f)) as h:
            text = h.read()
        for m in re.finditer(r"\bstatic\b[^;{}]*=\s*\[", text):
            body = text[m.end():text.index("}();", m.end())]
            assert "cudaFuncSetAttribute" not in body and "cudaOccupancy" not in body, (f, m.group(0))


PROGRAM = r"""
#include <cstdio>
#include <thread>
#include <vector>
#include "cfp_device.cuh"
int main() {
    cfp::OncePerDevice once;
    int calls[70] = {}, bad = 0;
    for (int round = 0; round < 3; ++round)
        for (int d = 0; d < 70; ++d) bad += once.run(d, [&] { return ++calls[d], 0; });
    for (int d = 0; d < 70; ++d) bad += calls[d] != (d < 64 ? 1 : 3);  // past the table: every time
    cfp::OncePerDevice fails;
    int n = 0;
    bad += fails.run(1, [&] { return ++n, 7; }) != 7;                  // a failure is not kept
    bad += fails.run(1, [&] { return ++n, 0; }) != 0;
    bad += fails.run(1, [&] { return ++n, 7; }) != 0 || n != 2;
    bad += fails.run(-1, [&] { return 3; }) != 3;
    cfp::OncePerDevice shared;
    std::atomic<int> ran{0};
    std::vector<std::thread> t;
    for (int q = 0; q < 8; ++q)
        t.emplace_back([&] { for (int d = 0; d < 64; ++d) shared.run(d, [&] { return ++ran, 0; }); });
    for (auto& x : t) x.join();
    bad += ran < 64 || ran > 8 * 64;
    std::printf("%d\n", bad);
    return bad != 0;
}
"""


def test_once_per_device(tmp_path):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no C++ compiler")
    src = tmp_path / "once.cpp"
    src.write_text(PROGRAM)
    exe = tmp_path / "once"
    subprocess.run([cxx, "-std=c++17", "-O1", "-pthread", "-I" + SRC, str(src), "-o", str(exe)], check=True)
    assert subprocess.run([str(exe)], capture_output=True, text=True).stdout == "0\n"
