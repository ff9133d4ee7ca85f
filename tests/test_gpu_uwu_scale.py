"""The weights-on-a-grid loss does not depend on the scale of the weights: rho0 = sum c^2 and the sums
over the constraints run in FP64, so weights whose squares lie below FP32's range give the loss of the
same weights at unit scale, and the gradient times the reciprocal scale. The scale is a power of two,
so that only what FP32 itself cannot hold of the spectrum (|rho|^2 of about 2^-127 at a quantum of
2^-149, 2e-7 relative) differs: the bars are those of the form's parity test."""

import numpy as np
import pytest

from paper_2305_15693_gb300 import inputs

from _parity import rel_l2

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    from paper_2305_15693_gb300 import _build
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    _build.build()


def test_loss_is_independent_of_the_weights_scale():
    import torch
    from paper_2305_15693_gb300 import fresco
    shape, scale = (4096, 2048), 2.0 ** -75      # (2^-75)^2 is half of FP32's smallest number
    g = inputs.rng(75)
    mask = inputs.ball_mask(12, 2)
    S0, W = 2.0 + g.random(len(mask)), 1e-5 * (0.5 + g.random(len(mask)))
    c = torch.from_numpy(2.0 * g.integers(0, 2, shape[::-1]).astype(np.float32) - 1.0).cuda()
    with fresco.Uwu(shape, mask, S0, W, "f32") as u:
        l1, g1 = u.loss_grad(c)
        l2, g2 = u.loss_grad(c * scale)
        torch.cuda.synchronize()
        l1, l2 = l1.item(), l2.item()
        g1, g2 = g1.double().cpu().numpy(), g2.double().cpu().numpy()
    assert np.isfinite(l1) and abs(l2 - l1) <= 1e-5 * l1
    assert rel_l2(g2 * scale, g1) <= 1e-4
