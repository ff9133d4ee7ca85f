"""FP64 2D spread on both sides of the rule that takes a tile's points by the whole block or by a thread
each: every point repeated eight times (and S0, W scaled so that the loss stays) has eight times the
points in every tile; rho is eight times as large, and each copy has an eighth of the gradient. Both
sides add the same windows: 1e-10 relative, as for the interpolation's rule."""

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


@pytest.mark.parametrize("width", [7, 8, 9, 10, 11, 12, 13])
def test_copies_of_points_add_up(width):
    import torch
    from paper_2305_15693_gb300 import fresco
    n, copies = 230, 8                   # (one or four tiles: 58 to 1840 points in each)
    g = inputs.rng(100 + width)
    mask = inputs.ball_mask(5, 2)
    S0, W = g.random(len(mask)), 0.5 + g.random(len(mask))
    pts = g.random((n, 2))
    out = []
    for c in (1, copies):
        x = torch.from_numpy(np.tile(pts, (c, 1))).cuda()
        with fresco.Plan(1.0, mask, c * S0, W / c ** 2, n * c, precision="f64",
                         width=width) as plan:
            loss, grad = plan.loss_grad(x)
            rho, _ = plan.rho_S()
            torch.cuda.synchronize()
            assert plan.status() == 0 and plan.launch_count() > 3
        out.append((loss.item(), rho.cpu().numpy() / c, c * grad.cpu().numpy().reshape(c, n, 2)))
    assert abs(out[0][0] - out[1][0]) <= 1e-10 * out[0][0]
    assert rel_l2(out[1][1], out[0][1]) <= 1e-10
    for copy in out[1][2]:
        assert rel_l2(copy, out[0][2][0]) <= 1e-10
