"""FP32 2D weights on a grid and points with free boundaries, with few and with very many constraints
per tile of the half plane: the rule that chooses between the half plane and the whole one (checked on
the CPU) and both forms against the oracle, at the bars of their parity tests."""

import os
import shutil
import subprocess

import numpy as np
import pytest

import oracle
from paper_2305_15693_gb300 import inputs

from _parity import rel_l2
from test_fastdiv_host import CSRC, ROOT, _cuda_include

PROGRAM = r"""
#include <cstdio>
#include "fresco_uwnu_tiles.h"
int main() {
    // fine grid, width, constraints
    const long c[][3] = {{128, 7, 8000}, {128, 7, 100000}, {224, 7, 10000}, {224, 7, 100000},
                         {320, 7, 100000}, {512, 7, 100000}, {512, 7, 1000000}, {800, 7, 1000000},
                         {2048, 7, 1000000}, {2048, 7, 100000000}, {30, 7, 100}};
    for (const auto &x : c) {
        const int nf[3] = {(int)x[0], (int)x[0], 1};
        std::printf("%d ", (int)fresco::half_plane_pays(nf, (int)x[1], x[2]));
    }
    return 0;
}
"""


def test_the_rule_follows_the_measurements(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    inc = _cuda_include()
    if not cxx or not inc:
        pytest.skip("needs a C++ compiler and the CUDA headers")
    src, exe = tmp_path / "half.cpp", tmp_path / "half"
    src.write_text(PROGRAM)
    subprocess.run([cxx, "-O2", "-std=c++17", "-I", os.path.join(ROOT, "include"), "-I", CSRC,
                    "-I", inc, str(src), "-o", str(exe)], check=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split()
    assert out == list("10100101111")


@pytest.mark.gpu
@pytest.mark.parametrize("shape,nk", [((64, 64), 8000), ((64, 64), 9000), ((33, 64), 7000),
                                      ((64, 33), 300)])
def test_weights_with_few_and_many_constraints_a_tile(shape, nk):
    import torch
    from paper_2305_15693_gb300 import fresco
    g = inputs.rng(nk + shape[0])
    c = g.standard_normal(int(np.prod(shape))).astype(np.float32)
    nu = (g.random((nk, 2)) - 0.5) * 0.9 * np.array(shape)
    S0, W = 0.2 * g.random(nk), 0.5 + g.random(nk)
    want_l, want_g, want_S, _ = oracle.weight_loss_grad_k(
        oracle.grid_points(shape), c.astype(np.float64), 2 * np.pi * nu, S0, W)
    with fresco.Uwnu(shape, nu, S0, W, "f32") as u:
        x = torch.from_numpy(c.reshape(shape[::-1])).cuda()
        loss, grad = u.loss_grad(x)
        l2, _ = u.loss_grad(x, want_grad=False)
        S = u.S().double().cpu().numpy()
    assert loss.item() == l2.item()
    assert rel_l2(S, want_S) <= 2e-5
    assert abs(loss.item() - want_l) <= 1e-5 * abs(want_l)
    assert rel_l2(grad.double().cpu().numpy().reshape(-1), want_g) <= 1e-4
