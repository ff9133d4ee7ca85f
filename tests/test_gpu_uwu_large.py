"""The largest weights-on-a-grid plans, on both sides of the rule that keeps the library's columns: a
few hundred weights that are not zero, so that the oracle's direct sums run over those cells alone, at
the bars of the form's parity test."""

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


@pytest.mark.parametrize("shape", [(16384, 16384), (16384, 8192), (2048, 16384)])
def test_sparse_weights_on_large_grids(shape):
    import torch
    from paper_2305_15693_gb300 import fresco
    g = inputs.rng(shape[1])
    mask = inputs.ball_mask(9, 2)
    S0, W = 0.3 * g.random(len(mask)), 0.5 + g.random(len(mask))
    cell = np.unique(g.integers(0, shape, (300, 2)), axis=0)
    v = g.standard_normal(len(cell)).astype(np.float32)
    want_l, want_g, _, _ = oracle.weight_loss_grad(cell / np.array(shape, dtype=np.float64),
                                                   v.astype(np.float64), mask, S0, W)
    at = torch.from_numpy(cell).cuda()
    c = torch.zeros(shape[::-1], device="cuda")
    c[at[:, 1], at[:, 0]] = torch.from_numpy(v).cuda()
    with fresco.Uwu(shape, mask, S0, W, "f32") as u:
        loss, grad = u.loss_grad(c)
        torch.cuda.synchronize()
        got = grad[at[:, 1], at[:, 0]].double().cpu().numpy()
    assert abs(loss.item() - want_l) <= 1e-5 * abs(want_l)
    assert rel_l2(got, want_g) <= 1e-4
