"""What a kernel is allowed on one device of a process says nothing of the
others (csrc/dsr_per_device.h): every device is asked, once, and keeps its own
answer. Plain C++ with a stand-in for the question, no GPU."""
import os
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1809_07444_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include "dsr_per_device.h"
int main() {
    static dsr_per_device fits;
    int asked[100] = {0};
    auto ask = [&](int d) { return fits.get(d, [&] { ++asked[d]; return d % 3 != 1; }); };
    for (int round = 0; round < 3; ++round)
        for (int d = 0; d < 70; ++d)
            if (ask(d) != (d % 3 != 1)) return 1;
    for (int d = 0; d < 70; ++d)
        if (asked[d] != (d < dsr_per_device::DEVICES ? 1 : 3)) return 2;
    return fits.get(-1, [] { return true; }) ? 0 : 3;
}
"""


def test_every_device_is_asked_once(tmp_path):
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    assert subprocess.run([str(exe)]).returncode == 0


def test_the_cluster_kernels_keep_no_answer_of_a_whole_process():
    for name in ("dsr_gol.cu", "dsr_wator.cu"):
        text = open(os.path.join(CSRC, name)).read()
        assert "static const bool" not in text and "static dsr_per_device fits;" in text
