"""Evaluations recorded in a CUDA graph by the caller: after a replay, reads of the plan's state (rho
and S) must belong to the replayed evaluation, as they do after an ordinary call."""

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


def test_first_read_of_a_small_plan_can_be_recorded():
    """A direct plan's first read of rho and S inside the recorded work: it allocates and uploads
    nothing, and a read that was recorded and never replayed leaves nothing behind for later ones."""
    import torch
    from paper_2305_15693_gb300 import fresco
    mask = inputs.ball_mask(9, 2)
    x = torch.from_numpy(inputs.uniform_points(300, 2, 3)).cuda()
    stream = torch.cuda.Stream()
    loss = torch.zeros((), dtype=torch.float64, device="cuda")
    rho = torch.zeros(len(mask), 2, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    with torch.cuda.stream(stream), fresco.Plan(1.0, mask, np.zeros(len(mask)), np.ones(len(mask)),
                                                300, precision="f64", stream=stream) as plan:
        fresco.fresco_forward(plan.handle, x, loss)
        stream.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            fresco.fresco_forward(plan.handle, x, loss)
            fresco.fresco_get_rho_S(plan.handle, rho, None)
        want, _ = plan.rho_S()          # (before any replay)
        graph.replay()
        stream.synchronize()
        assert plan.launch_count() > 0 and torch.equal(rho, want)


@pytest.mark.parametrize("mode", ["kderiv", "direct"])
@pytest.mark.parametrize("dim,width,precision", [(2, 7, "f32"), (2, 0, "f32"), (3, 7, "f32"),
                                                 (2, 13, "f64")])
def test_rho_after_a_replayed_evaluation_belongs_to_it(dim, width, precision, mode):
    """rho and S are read, the points change, the recorded evaluation is replayed, and rho and S are
    read again: they equal, bit for bit in FP32 (fixed-point spread, direct sums) and to rounding in
    FP64 (its sums in 2D follow the order the binning's atomics ran in), those after an ordinary
    evaluation of the same points."""
    import torch
    from paper_2305_15693_gb300 import fresco
    dt = torch.float64 if precision == "f64" else torch.float32
    n = 3000
    mask = inputs.ball_mask(19 if dim == 2 else 6, dim)
    S0, W = np.full(len(mask), 0.3), np.ones(len(mask))
    a, b = (torch.from_numpy(inputs.uniform_points(n, dim, s)).to("cuda", dt) for s in (1, 2))
    stream = torch.cuda.Stream()
    x, grad = a.clone(), torch.empty_like(a)
    loss = torch.zeros((), dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    with torch.cuda.stream(stream), fresco.Plan(1.0, mask, S0, W, n, precision=precision,
                                                width=width, grad_mode=mode,
                                                stream=stream) as plan:
        fresco.fresco_loss_grad(plan.handle, x, loss, grad)
        stream.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=stream):
            fresco.fresco_loss_grad(plan.handle, x, loss, grad)
        plan.loss_grad(a)
        plan.rho_S()
        x.copy_(b)
        graph.replay()
        rho, S = plan.rho_S()
        stream.synchronize()
        l1, g1 = loss.item(), grad.clone()
        l2, g2 = plan.loss_grad(b)
        rho2, S2 = plan.rho_S()
        stream.synchronize()
        assert plan.status() == 0
        l2 = l2.item()
    if precision == "f32":
        assert torch.equal(rho, rho2) and torch.equal(S, S2)
        assert l1 == l2 and torch.equal(g1, g2)
    else:
        torch.testing.assert_close(rho, rho2, rtol=0, atol=1e-9)
        torch.testing.assert_close(S, S2, rtol=0, atol=1e-9)
        assert abs(l1 - l2) <= 1e-12 * abs(l2)
        torch.testing.assert_close(g1, g2, rtol=0, atol=1e-9 * float(g2.abs().max()))
