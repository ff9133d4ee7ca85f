"""The pair term's cell rows against the oracle where they can go wrong: exactly three cells along
every axis (each row holds the whole axis, one cell of it wrapped), two cells along one axis only
(the general form), points on cell and box faces, a cell with most of the
points, a general exponent. Bars as for the other sizes: 1e-11 in FP64, 2e-5 in FP32."""

import numpy as np
import pytest

import oracle
from paper_2305_15693_gb300 import inputs

from _parity import rel_l2

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    from paper_2305_15693_gb300 import _build
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    _build.build()


CASES = {
    "three cells 2D": (2, 200, [1.0, 1.0], 0.33, 2.0, 0),
    "three cells 3D": (3, 300, [1.0, 1.1, 0.95], 0.31, 2.5, 0),
    "two cells along y": (3, 300, [2.0, 0.9, 2.0], 0.32, 2.0, 0),
    "many cells, a crowded one": (3, 900, [1.0, 1.0, 1.0], 0.09, 2.0, 400),
    "general exponent": (2, 500, [1.0, 1.3], 0.11, 3.25, 0),
}


@pytest.mark.parametrize("precision", ["f64", "f32"])
@pytest.mark.parametrize("name", sorted(CASES))
def test_cell_rows_match_oracle(name, precision):
    import torch
    from paper_2305_15693_gb300 import fresco
    dim, n, box, sigma, alpha, crowd = CASES[name]
    dt = np.float64 if precision == "f64" else np.float32
    g = inputs.rng(len(name))
    box = np.array(box)
    pts = g.random((n, dim)) * 3.0 - 1.0
    if crowd:
        pts[:crowd] = 0.512 + 0.02 * g.random((crowd, dim))
    pts[-4:] = np.arange(4)[:, None] / 4.0            # lattice sites, the box corner among them
    pts = np.ascontiguousarray((pts * box).astype(dt))
    e_o, g_o = oracle.pair_energy_grad(pts, sigma, 0.7, alpha, box=box)
    with fresco.PairTerm(box, dim, n, sigma, 0.7, alpha, precision) as pt:
        e, grad = pt.energy_grad(torch.from_numpy(pts).cuda())
        torch.cuda.synchronize()
    bar = 1e-11 if precision == "f64" else 2e-5
    assert e_o > 0
    assert abs(e.item() - e_o) <= bar * e_o
    assert rel_l2(grad.double().cpu().numpy(), g_o) <= bar
