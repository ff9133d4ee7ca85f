"""The device L-BFGS's vector forms (one cluster with 4 or 16 elements a thread, one launch per pair
and direction) against the numpy reference on the same plan's gradients, at the vector lengths where
the form changes and with short, long and odd histories: the losses of twelve iterations agree to
1e-9 relative (both sides run the same FP64 evaluations; only the order of the sums differs)."""

import numpy as np
import pytest

from paper_2305_15693_gb300 import inputs

from _lbfgs_ref import lbfgs as lbfgs_ref

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    from paper_2305_15693_gb300 import _build
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    _build.build()


@pytest.mark.parametrize("dim,n,history", [(2, 2, 4), (2, 33, 64), (2, 4096, 1), (2, 4097, 10),
                                           (2, 16384, 3), (2, 16385, 1), (2, 16385, 7),
                                           (3, 10922, 10), (3, 10923, 10)])
def test_iterates_follow_the_reference_at_every_vector_form(dim, n, history):
    import torch
    from paper_2305_15693_gb300 import fresco
    g = inputs.rng(n + history)
    mask = inputs.ball_mask(6 if dim == 2 else 3, dim)
    S0, W = 0.3 + g.random(len(mask)), np.ones(len(mask))
    x0 = g.random((n, dim))
    step = 0.1 * n ** (-1.0 / dim)
    with fresco.Plan(1.0, mask, S0, W, n, precision="f64") as plan:
        def fg(x):
            loss, grad = plan.loss_grad(torch.from_numpy(np.ascontiguousarray(x)).cuda())
            return loss.item(), grad.cpu().numpy()

        _, ref = lbfgs_ref(fg, x0, 12, m=history, max_step=step)
        pts = torch.from_numpy(x0).cuda()
        opt = fresco.LBFGS(plan, history=history, max_step=step)
        trace = [opt.run(pts, 1)["loss"] for _ in range(12)]
        opt.close()
    k = min(len(ref) - 1, 12)
    assert k >= 2
    np.testing.assert_allclose(trace[:k], ref[1:k + 1], rtol=1e-9, atol=1e-24)
