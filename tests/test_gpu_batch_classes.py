"""Ensembles of many size classes: more than one launch takes, and classes whose rows or columns need
far more shared memory than the others'. Every instance against the oracle; targets are zero, so the
loss has no cancellation and the bars are the kernel tolerance's."""

import numpy as np
import pytest

import oracle

from _parity import TOL, rel_l2

pytestmark = pytest.mark.gpu


def _instances(big):
    rng = np.random.default_rng(5)
    kmax = [(kx, ky) for kx in (5, 10, 20, 40) for ky in (5, 10, 20, 40, 80)]
    if big:
        kmax = kmax[::6] + [(2900, 9), (9, 1400)]
    out = []
    for kx, ky in kmax:
        m = np.stack([rng.integers(-kx, kx + 1, 60), rng.integers(-ky, ky + 1, 60)], 1)
        m = np.concatenate([m, [[kx, ky], [kx, 1 - ky], [0, ky], [kx, 0]]])
        m = np.unique(m[np.any(m != 0, 1)], axis=0).astype(np.int32)
        # points on a 2^-12 lattice: their places on every grid are exact in FP32, which would
        # otherwise add |k| x 2^-24 of phase to the kernel's own error
        n = int(rng.integers(1, 700))
        out.append((1.0, m, rng.integers(-2048, 2048, (n, 2)) / 4096.0))
    return out


@pytest.mark.parametrize("grad_mode", ["kderiv", "direct"])
@pytest.mark.parametrize("big", [False, True])
def test_many_size_classes(grad_mode, big):
    import torch
    from paper_2305_15693_gb300 import fresco
    inst = _instances(big)
    masks = [m for _, m, _ in inst]
    zero = [np.zeros(len(m)) for m in masks]
    one = [np.ones(len(m)) for m in masks]
    pts = np.concatenate([p for _, _, p in inst]).astype(np.float32)
    with fresco.Batch([b for b, _, _ in inst], [len(p) for _, _, p in inst], masks, zero, one,
                      precision="f32", grad_mode=grad_mode) as b:
        losses, grad = b.loss_grad(torch.from_numpy(pts).cuda())
        only, _ = b.loss_grad(torch.from_numpy(pts).cuda(), want_grad=False)
        torch.cuda.synchronize()
        assert b.status() == fresco.FRESCO_OK
        first = b.first
        losses, grad, only = losses.cpu().numpy(), grad.double().cpu().numpy(), only.cpu().numpy()
    assert np.array_equal(losses, only)
    for i, (box, m, _) in enumerate(inst):
        p = pts[first[i]:first[i + 1]].astype(np.float64)
        l_o, g_o, _, _ = oracle.loss_grad(p, m, zero[i], one[i], box=box)
        assert abs(losses[i] - l_o) <= TOL["f32"]["loss"] * abs(l_o), i
        if len(p) > 1:
            assert rel_l2(grad[first[i]:first[i + 1]], g_o) <= TOL["f32"]["grad"], i
