"""Kernel attributes are raised on every device a process uses, not on its first one: the host class on a
fake of the device, compiled here (a second GPU would see the default 48 KB of shared memory and
refuse the larger launches), and its use by every file that raises them."""
import os
import re
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2306_06007_gb300", "csrc")

PROGRAM = r"""
#include "per_device.h"
#include <cstdio>
#include <stdexcept>
int main() {
    static hvox::OncePerDevice once, other;
    int calls[300] = {0}, bad = 0;
    for (int round = 0; round < 3; ++round)
        for (int dev : {0, 1, 63, 64, 255, 299}) once.run(dev, [&] { ++calls[dev]; });
    for (int dev : {0, 1, 63, 64, 255}) bad += calls[dev] != 1;
    bad += calls[299] != 3;                       // beyond the table: every time
    try { other.run(2, [] { throw std::runtime_error("refused"); }); } catch (const std::exception &) {}
    other.run(2, [&] { ++calls[2]; });            // a failed one is tried again
    bad += calls[2] != 1;
    std::printf("%d\n", bad);
    return bad;
}
"""


@pytest.mark.skipif(shutil.which("g++") is None, reason="needs a C++ compiler")
def test_once_per_device(tmp_path):
    (tmp_path / "t.cpp").write_text(PROGRAM)
    subprocess.run(["g++", "-std=c++17", "-I", CSRC, str(tmp_path / "t.cpp"), "-o", str(tmp_path / "t")], check=True)
    assert subprocess.run([str(tmp_path / "t")], capture_output=True, text=True, check=True).stdout.strip() == "0"


@pytest.mark.parametrize("name", ["k_direct.cu", "k_cfft.cu", "k_dffft.cu", "k_nufft.cu"])
def test_attributes_are_raised_per_device(name):
    src = open(os.path.join(CSRC, name)).read()
    assert "cudaFuncSetAttribute" in src and "OncePerDevice" in src
    assert not re.search(r"once_flag|call_once", src)
