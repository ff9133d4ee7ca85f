"""CPU check of the length of the 3D column spread's segments (z_segment in csrc/fresco_internal.h):
never longer than the grid has tiles, a whole number of tiles, and in the fixed-point (FP32) spread
never more than six, because the tiles of a segment share the scale of its most crowded tile."""

import os
import shutil
import subprocess

import pytest

from test_fastdiv_host import CSRC, ROOT, _cuda_include

PROGRAM = r"""
#include <cstdio>
#include "fresco_internal.h"
int main() {
    long bad = 0, checked = 0;
    for (int xy = 1; xy <= 80; ++xy)
        for (int z = 1; z <= 120; ++z)
            for (int per_sm = 0; per_sm <= 4; ++per_sm)
                for (int fixed = 0; fixed < 2; ++fixed, ++checked) {
                    const int nb[3] = {xy, (xy + 1) / 2, z};
                    const int s = fresco::z_segment(nb, per_sm, fixed != 0);
                    if (s < 1 || s > z || s > (fixed ? 6 : 16) || (z > 1 && s < 2)) ++bad;
                }
    std::printf("%ld %ld\n", bad, checked);
    return 0;
}
"""


def test_segment_lengths(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    inc = _cuda_include()
    if not cxx or not inc:
        pytest.skip("needs a C++ compiler and the CUDA headers")
    src, exe = tmp_path / "zseg.cpp", tmp_path / "zseg"
    src.write_text(PROGRAM)
    subprocess.run([cxx, "-O2", "-std=c++17", "-I", os.path.join(ROOT, "include"), "-I", CSRC,
                    "-I", inc, str(src), "-o", str(exe)], check=True)
    bad, checked = map(int, subprocess.run([str(exe)], check=True, capture_output=True,
                                           text=True).stdout.split())
    assert checked == 80 * 120 * 5 * 2 and bad == 0
