"""Weight and gradient arrays of the weights-on-a-grid form that are views at offsets of a larger
buffer, as a program has them that keeps its weights in one flat parameter vector: the gradient
anywhere a float may lie, the weights on a boundary of two floats, and the error for weights that are
not, the same whether a grid runs the library's own transforms or cuFFT's. Checked against the oracle
at the bars of the form's parity test; nothing outside the gradient's own cells is written."""

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


SHAPES = [((64, 22), 9), ((12, 100), 5), ((64, 20), 9)]   # (22 = 2 x 11 keeps cuFFT)


@pytest.mark.parametrize("off_c,off_g", [(0, 0), (0, 1), (2, 3), (2, 2)])
@pytest.mark.parametrize("shape,K", SHAPES)
def test_weights_and_gradient_at_offsets(shape, K, off_c, off_g):
    import torch
    from paper_2305_15693_gb300 import fresco
    g = inputs.rng(shape[0])
    n = int(np.prod(shape))
    mask = inputs.ball_mask(K, 2)
    c = g.standard_normal(n).astype(np.float32)
    S0, W = 0.3 * g.random(len(mask)), 0.2 + g.random(len(mask))
    want_l, want_g, _, _ = oracle.weight_loss_grad(oracle.grid_points(shape), c.astype(np.float64),
                                                   mask, S0, W)
    flat = torch.zeros(n + 8, device="cuda")
    flat[off_c:off_c + n] = torch.from_numpy(c).cuda()
    out = torch.full((n + 8,), 7.0, device="cuda")
    loss = torch.zeros((), dtype=torch.float64, device="cuda")
    with fresco.Uwu(shape, mask, S0, W, "f32") as u:
        fresco.fresco_uwu_loss_grad(u.handle, flat[off_c:off_c + n], loss, out[off_g:off_g + n])
        l2, _ = u.loss_grad(flat[off_c:off_c + n].view(shape[::-1]), want_grad=False)
        torch.cuda.synchronize()
    out = out.cpu().numpy()
    assert np.all(out[:off_g] == 7.0) and np.all(out[off_g + n:] == 7.0)
    assert l2.item() == loss.item()
    assert abs(loss.item() - want_l) <= 1e-5 * abs(want_l)
    assert rel_l2(out[off_g:off_g + n].astype(np.float64), want_g) <= 1e-4


@pytest.mark.parametrize("shape,K", SHAPES)
def test_weights_at_an_odd_offset_are_refused(shape, K):
    import torch
    from paper_2305_15693_gb300 import fresco
    mask = inputs.ball_mask(K, 2)
    n = int(np.prod(shape))
    flat = torch.ones(n + 1, device="cuda")
    with fresco.Uwu(shape, mask, np.zeros(len(mask)), np.ones(len(mask)), "f32") as u:
        with pytest.raises(fresco.FrescoError) as e:
            u.loss_grad(flat[1:].view(shape[::-1]))
        assert e.value.status == fresco.FRESCO_ERR_CUFFT
        u.loss_grad(flat[:n].view(shape[::-1]))
        torch.cuda.synchronize()
