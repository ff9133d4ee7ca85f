"""CPU check of the slots per tile of the direct binning form (direct_tile_capacity in
csrc/fresco_internal.h): points drawn uniformly over the cells they lie in (the whole grid, or a part
of it as in the free-boundary form, whose grid has spare cells around the box) never overflow a tile."""

import os
import shutil
import subprocess

import pytest

from test_fastdiv_host import CSRC, ROOT, _cuda_include

PROGRAM = r"""
#include <cstdio>
#include <cstdint>
#include <vector>
#include "fresco_internal.h"
using namespace fresco;
static uint64_t s = 88172645463325252ULL;
static double uni() { s ^= s << 13; s ^= s >> 7; s ^= s << 17; return (double)(s >> 11) / 9007199254740992.0; }
int main() {
    long over = 0, checked = 0;
    const int cases[][4] = {   // dim, grid, tile, cells the points lie in
        {2, 112, 28, 100}, {2, 210, 30, 200}, {2, 320, 32, 300}, {2, 420, 30, 400}, {2, 1620, 30, 1600},
        {2, 210, 30, 210}, {3, 40, 10, 30}, {3, 70, 10, 60}, {3, 140, 14, 120}, {3, 140, 14, 140},
        {2, 64, 32, 20}};
    for (const auto &c : cases) {
        Geom g{};
        g.dim = c[0];
        g.n_tiles = 1;
        double extent[3] = {1, 1, 1};
        for (int a = 0; a < 3; ++a) {
            g.nf[a] = a < g.dim ? c[1] : 1;
            g.nb[a] = a < g.dim ? c[1] / c[2] : 1;
            g.tmax[a] = a < g.dim ? c[2] : 1;
            g.n_tiles *= g.nb[a];
            if (a < g.dim) extent[a] = c[3];
        }
        g.n_points = 400000;
        const int cap = direct_tile_capacity(g, extent);
        if (!cap) continue;   // too many slots: the compact form from the start
        std::vector<int> n((size_t)g.n_tiles, 0);
        for (int64_t j = 0; j < g.n_points; ++j) {
            int t = 0;
            for (int a = g.dim - 1; a >= 0; --a) {   // centred on cell 0, wrapped
                const int x = (int)((uni() - 0.5) * c[3] + c[1]) % c[1];
                t = t * g.nb[a] + x / c[2];
            }
            ++n[(size_t)t];
        }
        for (int v : n) over += v > cap;
        checked += g.n_tiles;
    }
    std::printf("%ld %ld\n", over, checked);
    return 0;
}
"""


def test_uniform_points_never_overflow(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    inc = _cuda_include()
    if not cxx or not inc:
        pytest.skip("needs a C++ compiler and the CUDA headers")
    src, exe = tmp_path / "cap.cpp", tmp_path / "cap"
    src.write_text(PROGRAM)
    subprocess.run([cxx, "-O2", "-std=c++17", "-I", os.path.join(ROOT, "include"), "-I", CSRC,
                    "-I", inc, str(src), "-o", str(exe)], check=True)
    over, checked = map(int, subprocess.run([str(exe)], check=True, capture_output=True,
                                            text=True).stdout.split())
    assert checked > 4000 and over == 0
