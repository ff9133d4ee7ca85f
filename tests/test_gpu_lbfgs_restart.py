"""The device L-BFGS where the stored pairs give no descent direction: it restarts from the steepest
descent, on both vector forms, without an evaluation at a point along the dropped direction. Points
that no evaluation was asked for must not reach the plan (its error word is latched by a coordinate
that is not finite), and the report counts every evaluation."""

import numpy as np
import pytest

from paper_2305_15693_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    from paper_2305_15693_gb300 import _build
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    _build.build()


@pytest.mark.parametrize("n", [64, 17000])
def test_degenerate_pairs_restart_without_a_stray_evaluation(n):
    """Points within 1e-158 of the origin and S0 = 2 N: the loss is quadratic in the points with the
    gradient u c, u = x - mean(x), c = 4 W N sum_n (2 pi n_x)^2, so that with c = 1/2 every accepted
    steepest-descent step halves u. s.y is about 1e-315, its reciprocal is infinite and the next
    direction is not a number: every iteration after the first restarts. (n = 17000: vectors longer
    than one cluster's registers.) The sums at rounding of u: 1e-9 relative is ample."""
    import torch
    from paper_2305_15693_gb300 import fresco
    mask = inputs.ball_mask(2, 2)
    c = 0.5
    W = c / (4.0 * n * np.sum((2.0 * np.pi * mask[:, 0]) ** 2))
    x0 = 1e-158 * (2.0 * inputs.rng(n).random((n, 2)) - 1.0)
    x = torch.from_numpy(x0).cuda()
    with fresco.Plan(1.0, mask, np.full(len(mask), 2.0 * n), np.full(len(mask), W), n,
                     precision="f64") as plan:
        assert plan.status() == 0
        plan.loss_grad(x)
        per_call = plan.launch_count()
        opt = fresco.LBFGS(plan, max_step=0.1)
        rep = opt.run(x, 6)
        opt.close()
        assert plan.status() == 0
        assert plan.launch_count() == per_call * (1 + rep["evaluations"])
    assert rep["iterations"] == 6 and rep["evaluations"] == 7 and rep["status"] == 3
    mean = x0.mean(0)
    np.testing.assert_allclose(x.cpu().numpy() - mean, (x0 - mean) * 0.5 ** 6, rtol=0,
                               atol=1e-9 * 1e-158)


def test_zero_gradient_stops_before_any_trial():
    """One point at the origin has S = 1 exactly; with S0 = 1 its gradient is exactly zero, and the
    run ends with the start's evaluation (three launches) alone."""
    import torch
    from paper_2305_15693_gb300 import fresco
    mask = inputs.ball_mask(3, 2)
    x = torch.zeros(1, 2, dtype=torch.float64, device="cuda")
    with fresco.Plan(1.0, mask, np.ones(len(mask)), np.ones(len(mask)), 1,
                     precision="f64") as plan:
        opt = fresco.LBFGS(plan, max_step=0.1)
        rep = opt.run(x, 5)
        opt.close()
        assert plan.launch_count() == 3
    assert rep["evaluations"] == 1 and rep["iterations"] == 0 and rep["status"] == 1
