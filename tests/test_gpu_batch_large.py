"""FP32 ensembles on both sides of the rule for the library's own transforms (few size classes with
very many cells keep cuFFT): losses and gradients of every instance against single plans of the same
problem on the same kernel width, at the bars of the parity tests."""

import numpy as np
import pytest

from paper_2305_15693_gb300 import inputs

from _parity import TOL, rel_l2

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    from paper_2305_15693_gb300 import _build
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    _build.build()


@pytest.mark.parametrize("mode", ["kderiv", "direct"])
@pytest.mark.parametrize("Ks", [(510,) * 4, (250,) * 3, (250, 510, 30, 510, 510),
                                (250, 510, 30, 510, 510, 510, 510)])
def test_instances_match_single_plans(Ks, mode):
    """Grids of 2048^2 (K = 510), 1024^2 (250) and 128^2 (30): 1.7e7 and 3.1e6 cells in one class,
    1.4e7 and 2.2e7 in three."""
    import torch
    from paper_2305_15693_gb300 import fresco
    g = inputs.rng(len(Ks))
    n = [3000 + 500 * i for i in range(len(Ks))]
    masks = [m[g.permutation(len(m))[:4000]] for m in (inputs.ball_mask(K, 2) for K in Ks)]
    masks = [np.vstack([m, [[K, 0], [0, K]]]).astype(np.int32) for m, K in zip(masks, Ks)]
    S0s = [g.random(len(m)) for m in masks]
    Ws = [0.5 + g.random(len(m)) for m in masks]
    pts = torch.from_numpy(g.random((sum(n), 2)).astype(np.float32)).cuda()
    with fresco.Batch([1.0] * len(Ks), n, masks, S0s, Ws, "f32", width=7, grad_mode=mode) as b:
        for _ in range(2):
            losses, grad = b.loss_grad(pts)
        torch.cuda.synchronize()
        assert b.status() == 0
        parts, got = b.split(grad), losses.cpu().numpy()
        for i, x in enumerate(b.split(pts)):
            with fresco.Plan(1.0, masks[i], S0s[i], Ws[i], n[i], width=7, grad_mode=mode) as p:
                loss, want = p.loss_grad(x.contiguous())
                torch.cuda.synchronize()
            assert abs(got[i] - loss.item()) <= 2 * TOL["f32"]["loss"] * loss.item()
            assert rel_l2(parts[i].cpu().numpy(), want.cpu().numpy()) <= 2 * TOL["f32"]["grad"]
