"""FP64 3D interpolation on both sides of the rule that gives a tile's points a warp or a thread each:
every point repeated eight times (and S0, W scaled so that the loss stays) has eight times the points
in every tile and must give each copy an eighth of the gradient. Both sides evaluate the same sums, so
they agree to FP64 rounding whatever the kernel's width: 1e-10 relative, 1e5 times the unit roundoff
for sums of some hundred terms of either sign that cancel to a part of their size."""

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


@pytest.mark.parametrize("K,n", [(6, 900), (14, 9000)])   # (fewer tiles than SMs, and more)
@pytest.mark.parametrize("mode", ["direct", "kderiv"])
@pytest.mark.parametrize("width", [2, 3, 4, 5, 6, 7, 8, 10, 12])
def test_copies_of_points_share_the_gradient(width, mode, K, n):
    import torch
    from paper_2305_15693_gb300 import fresco
    copies = 8
    g = inputs.rng(width)
    mask = inputs.ball_mask(K, 3)
    S0, W = g.random(len(mask)), 0.5 + g.random(len(mask))
    pts = g.random((n, 3))
    out = []
    for c in (1, copies):
        x = torch.from_numpy(np.tile(pts, (c, 1))).cuda()
        with fresco.Plan(1.0, mask, c * S0, W / c ** 2, n * c, precision="f64", width=width,
                         grad_mode=mode) as plan:
            loss, grad = plan.loss_grad(x)
            torch.cuda.synchronize()
            assert plan.status() == 0 and plan.launch_count() > 3
        out.append((loss.item(), c * grad.cpu().numpy().reshape(c, n, 3)))
    assert abs(out[0][0] - out[1][0]) <= 1e-10 * out[0][0]
    for copy in out[1][1]:
        assert rel_l2(copy, out[0][1][0]) <= 1e-10
