"""FP64 tiles whose points the block takes together (spread: residue-owned cells; 3D
interpolation: one warp per point) against the oracle, on both sides of their rules: kernels
narrower and at least eight cells wide, sparse tiles and tiles of more than 128 points, ragged
sizes and boxes, column segments that end inside the grid. The bars scale the FP64 ones (10, 100
and 1000 times the plan tolerance for rho, loss and gradient) to the tolerance of each width."""

import numpy as np
import pytest

from paper_2305_15693_gb300 import inputs

from _parity import compare

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    from paper_2305_15693_gb300 import _build
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    _build.build()


@pytest.mark.parametrize("mode", ["direct", "kderiv"])
@pytest.mark.parametrize("dim,tol,width", [(2, 1e-12, 13), (2, 3e-8, 8), (3, 1e-12, 13),
                                           (3, 1e-11, 12), (3, 3e-8, 8), (3, 1e-6, 7)])
def test_block_taken_points_match_oracle(dim, tol, width, mode):
    g = inputs.rng(500 + 10 * dim + width)
    K = 21 if dim == 2 else 7
    n_bg, n_cl = (1501, 700) if dim == 2 else (1203, 450)
    box = np.linspace(0.9, 1.2, dim)
    pts = np.vstack([g.random((n_bg, dim)) * 3.0 - 1.0,
                     0.41 + 0.004 * g.standard_normal((n_cl, dim))]) * box
    mask = inputs.ball_mask(K, dim)
    S0, W = g.random(mask.shape[0]), 0.5 + g.random(mask.shape[0])
    err = compare(pts, mask, S0, W, box=box, precision="f64", tol=tol,
                  grad_mode=0 if mode == "direct" else 1)
    assert err["status"] == 0 and err["info"]["width"] <= width
    e = max(tol, 1e-12)
    assert err["rho"] <= 10 * e and err["loss"] <= 100 * e and err["grad"] <= 1000 * e, err
