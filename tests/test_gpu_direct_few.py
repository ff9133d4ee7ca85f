"""Small plans of few points and many wavevectors on both sides of the rule that chooses between direct
sums and the NUFFT: the form taken (its launches) and rho, loss and gradient against the oracle at the
parity tests' bars."""

import numpy as np
import pytest

import oracle
from paper_2305_15693_gb300 import inputs

from _parity import TOL, rel_l2

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    from paper_2305_15693_gb300 import _build
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    _build.build()


def _mask(form, K):
    if form in ("disk", "ball"):
        return inputs.ball_mask(K, 2 if form == "disk" else 3)
    if form == "sparse":
        m = inputs.rng(K).integers(-K, K + 1, (30, 2))
    else:   # strip
        a, b = np.meshgrid(np.arange(-K, K + 1), np.arange(-1, 2))
        m = np.stack([a.ravel(), b.ravel()], 1)
    return np.ascontiguousarray(m[np.any(m != 0, axis=1)].astype(np.int32))


@pytest.mark.parametrize("form,n,K,precision,direct", [
    ("disk", 1, 90, "f32", True), ("disk", 1, 200, "f32", False), ("disk", 300, 60, "f32", True),
    ("disk", 100, 300, "f32", False), ("disk", 150, 130, "f32", False),
    ("disk", 100, 50, "f64", True), ("disk", 50, 100, "f64", False),
    ("disk", 2000, 50, "f64", False), ("sparse", 10, 500, "f32", True),
    ("sparse", 10, 500, "f64", True), ("strip", 20, 2000, "f32", False), ("strip", 20, 3000, "f32", False),
    ("strip", 20, 100, "f32", True), ("disk", 12000, 10, "f64", True),
    ("disk", 100000, 6, "f32", True), ("ball", 3000, 8, "f64", True), ("ball", 4000, 10, "f32", True)])
def test_form_and_parity(form, n, K, precision, direct):
    import torch
    from paper_2305_15693_gb300 import fresco
    g = inputs.rng(n + K)
    dt = np.float64 if precision == "f64" else np.float32
    mask = _mask(form, K)
    pts = g.random((n, mask.shape[1])).astype(dt)
    S0, W = 0.3 * g.random(len(mask)), 0.5 + g.random(len(mask))
    want_l, want_g, _, want_rho = oracle.loss_grad(pts, mask, S0, W)
    with fresco.Plan(1.0, mask, S0, W, n, precision=precision) as plan:
        loss, grad = plan.loss_grad(torch.from_numpy(pts).cuda())
        assert (plan.launch_count() == 3) == direct
        rho, _ = plan.rho_S()
        torch.cuda.synchronize()
        assert plan.status() == 0
        held = plan.info["device_bytes"]
    assert held < 1.2e8
    rho = (rho[:, 0].double() + 1j * rho[:, 1].double()).cpu().numpy()
    assert rel_l2(rho, want_rho) <= TOL[precision]["rho"]
    assert abs(loss.item() - want_l) <= TOL[precision]["loss"] * abs(want_l)
    # (one point feels no force: its gradient is held against the terms that cancel in it)
    terms = 4.0 * W * np.abs(1.0 - S0) * 2.0 * np.pi * np.linalg.norm(mask, axis=1)
    scale = np.linalg.norm(terms) if n == 1 else np.linalg.norm(want_g)
    assert np.linalg.norm(grad.double().cpu().numpy() - want_g) <= TOL[precision]["grad"] * scale
