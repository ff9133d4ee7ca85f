"""Small plans run as direct sums; the same problem with the kernel width given runs the NUFFT. Both
forms against the oracle over everything a plan accepts: 2D and 3D, both precisions and gradient
modes, masks that are one-sided, sparse, repeated or partly of zero weight, boxes that are not cubes,
points outside the box, the smallest problems, and sizes on both sides of the rule. The direct sums
carry only the arithmetic's rounding: FP64 within 1e-12 (rho) of the oracle, FP32 within the bars of
the NUFFT path."""

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


def _evaluate(pts, mask, S0, W, box, precision, mode, width, host=False):
    import torch
    from paper_2305_15693_gb300 import fresco
    with fresco.Plan(box, mask, S0, W, pts.shape[0], precision=precision, grad_mode=mode,
                     width=width) as plan:
        x = torch.from_numpy(pts).cuda()
        loss, grad = plan.loss_grad(x)
        rho, S = plan.rho_S()
        n0 = plan.launch_count()
        plan.forward(x)
        go = torch.tensor(-2.0, dtype=torch.float64, device="cuda")
        g2 = plan.backward(go)
        launches = plan.launch_count() - n0
        gh = np.empty_like(pts)
        lh = plan.loss_grad_host(pts, gh)
        torch.cuda.synchronize()
        assert plan.status() == 0
        rho = (rho[:, 0].double() + 1j * rho[:, 1].double()).cpu().numpy()
        out = (loss.item(), grad.double().cpu().numpy(), rho, S.double().cpu().numpy())
        eps = 1e-12 if precision == "f64" else 1e-5
        assert rel_l2(g2.double().cpu().numpy(), -2.0 * out[1]) <= eps
        assert abs(lh - out[0]) <= eps * abs(out[0]) and rel_l2(gh, out[1]) <= eps
    return out, launches


def _masks(dim):
    g = inputs.rng(12 + dim)
    ball = inputs.ball_mask(11 if dim == 2 else 5, dim)
    half = ball[inputs.half_space(ball)]
    few = np.array([[37, -2, 3], [0, 5, -7], [-1, 0, 4], [4, 0, 0], [0, 0, -9], [0, -3, 0]],
                   dtype=np.int32)[:, :dim]
    few = few[np.any(few != 0, axis=1)]
    repeated = np.vstack([half, -half[::2], half[::3]])
    return {"ball": ball, "one-sided": -half, "sparse": few, "repeated": repeated,
            "shuffled": ball[g.permutation(len(ball))], "single": few[:1]}


@pytest.mark.parametrize("precision", ["f64", "f32"])
@pytest.mark.parametrize("dim", [2, 3])
@pytest.mark.parametrize("form", ["ball", "one-sided", "sparse", "repeated", "shuffled", "single"])
def test_direct_sums_and_nufft_match_the_oracle(form, dim, precision):
    g = inputs.rng(len(form) + dim)
    dt = np.float64 if precision == "f64" else np.float32
    box = np.linspace(1.3, 0.8, dim)
    mask = np.ascontiguousarray(_masks(dim)[form])
    n = 1 if form == "single" else 777
    pts = np.ascontiguousarray(((3.0 * g.random((n, dim)) - 1.0) * box).astype(dt))
    S0, W = g.random(len(mask)), 0.2 + g.random(len(mask))
    if len(mask) > 10:
        W[::7] = 0.0
    mode = "direct" if len(form) % 2 else "kderiv"
    want_l, want_g, want_S, want_rho = oracle.loss_grad(pts, mask, S0, W, box=box)
    for width in (0, 13 if precision == "f64" else 7):
        (loss, grad, rho, S), launches = _evaluate(pts, mask, S0, W, box, precision, mode, width)
        assert (launches == 3) == (width == 0)
        bar = dict(TOL[precision])
        if width == 0 and precision == "f64":
            bar = {"rho": 1e-12, "loss": 1e-11, "grad": 1e-11}
        assert rel_l2(rho, want_rho) <= bar["rho"]
        assert rel_l2(S, want_S) <= 4 * bar["rho"]
        # d loss = 2 sum W (S - S0) dS with dS <= 2 rho S, the conditioning a single wavevector
        # does not average away
        cond = 4 * bar["rho"] * np.sum(W * np.abs(want_S - S0) * want_S)
        assert abs(loss - want_l) <= max(bar["loss"] * abs(want_l), cond)
        assert rel_l2(grad, want_g) <= bar["grad"] or np.linalg.norm(want_g) < 1e-9


@pytest.mark.parametrize("dim,n,K,precision", [
    (2, 7, 3, "f32"), (2, 4863, 30, "f32"), (2, 4865, 31, "f32"), (2, 3000, 100, "f32"),
    (3, 5001, 9, "f32"), (3, 153, 12, "f64"), (2, 2600, 29, "f64"), (2, 31, 64, "f64")])
def test_sizes_across_blocks_and_the_rule(dim, n, K, precision):
    """Chunks of one and many points, several staged groups of coefficients, 8 and 32 points per
    gradient block, and one size beyond the rule (n = 3000, K = 100), which runs the NUFFT."""
    g = inputs.rng(n + K)
    dt = np.float64 if precision == "f64" else np.float32
    pts = g.random((n, dim)).astype(dt)
    mask = inputs.ball_mask(K, dim)
    S0, W = g.random(len(mask)), np.ones(len(mask))
    want_l, want_g, _, want_rho = oracle.loss_grad(pts, mask, S0, W)
    (loss, grad, rho, _), launches = _evaluate(pts, mask, S0, W, 1.0, precision, "kderiv", 0)
    bar = TOL[precision]
    assert (launches == 3) == (K != 100)
    assert rel_l2(rho, want_rho) <= bar["rho"] and rel_l2(grad, want_g) <= bar["grad"]
    assert abs(loss - want_l) <= bar["loss"] * abs(want_l)


def test_loose_tolerance_and_given_tiles_keep_the_nufft():
    import torch
    from paper_2305_15693_gb300 import fresco
    pts = torch.rand(500, 2, device="cuda")
    mask = inputs.ball_mask(8, 2)
    S0, W = np.zeros(len(mask)), np.ones(len(mask))
    for kw in ({"tol": 1e-3}, {"tile": (32, 32)}, {"width": 5}):
        with fresco.Plan(1.0, mask, S0, W, 500, **kw) as plan:
            plan.loss_grad(pts)
            assert plan.launch_count() > 3


def test_direct_plan_drives_the_tile_ordered_solver():
    """A solver that asks for tile order on a direct plan keeps the caller's order."""
    import torch
    from paper_2305_15693_gb300 import fresco
    pts0 = inputs.uniform_points(900, 2, 3)
    mask = inputs.ball_mask(17, 2)
    S0, W = np.zeros(len(mask)), np.ones(len(mask))
    got = []
    for tile_order in (False, True):
        pts = torch.from_numpy(pts0).cuda()
        with fresco.Plan(1.0, mask, S0, W, 900, precision="f64") as plan:
            opt = fresco.LBFGS(plan, tile_order=tile_order)
            got.append((opt.run(pts, 15)["loss"], pts.cpu().numpy()))
            opt.close()
    assert got[0][0] == got[1][0]
    np.testing.assert_array_equal(got[0][1], got[1][1])
