"""The NUFFT path of single plans (the kernel width is given, so that small problems do not run as
direct sums) against the oracle: transforms of many lengths on both sides of the rule for the
library's own kernels, grids that are not square, tiles narrower and wider than the kernel (the ring
fold by passes or by gathering), and binning after a tile overflowed. Half-plane transforms of the
weights-on-a-grid forms at their edges. Bars: the ones of the parity tests."""

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


def _check(pts, mask, precision="f32", mode="kderiv", width=7, box=1.0, tile=None, twice=False):
    import torch
    from paper_2305_15693_gb300 import fresco
    dt = np.float64 if precision == "f64" else np.float32
    pts = np.ascontiguousarray(pts.astype(dt))
    g = inputs.rng(len(mask))
    S0, W = g.random(len(mask)), 0.5 + g.random(len(mask))
    want_l, want_g, _, want_rho = oracle.loss_grad(pts, mask, S0, W, box=box)
    with fresco.Plan(box, mask, S0, W, pts.shape[0], precision=precision, width=width, tile=tile,
                     grad_mode=mode) as plan:
        x = torch.from_numpy(pts).cuda()
        for _ in range(2 if twice else 1):
            loss, grad = plan.loss_grad(x)
        rho, _ = plan.rho_S()
        rho2, _ = plan.rho_S()
        g2 = plan.backward()                     # the coefficients outlive a read of rho
        torch.cuda.synchronize()
        assert plan.status() == 0
        info = plan.info
    assert torch.equal(rho, rho2) and torch.equal(grad, g2)
    rho = (rho[:, 0].double() + 1j * rho[:, 1].double()).cpu().numpy()
    bar = TOL[precision]
    assert rel_l2(rho, want_rho) <= bar["rho"]
    assert abs(loss.item() - want_l) <= bar["loss"] * abs(want_l)
    assert rel_l2(grad.double().cpu().numpy(), want_g) <= bar["grad"]
    return info


def _box_mask(kx, ky, n, seed):
    """n wavevectors of the rectangle |n_x| <= kx, |n_y| <= ky, its corners among them."""
    g = inputs.rng(seed)
    m = np.stack([g.integers(-kx, kx + 1, n), g.integers(-ky, ky + 1, n)], 1)
    m[:3] = [[kx, ky], [-kx, ky], [0, ky]]
    m = m[np.any(m != 0, axis=1)]
    return np.ascontiguousarray(m.astype(np.int32))


@pytest.mark.parametrize("mode", ["kderiv", "direct"])
@pytest.mark.parametrize("kx,ky", [(3, 4), (4, 11), (6, 17), (12, 3), (15, 20), (24, 31), (31, 33),
                                   (52, 9), (8, 110), (95, 97), (170, 121), (260, 280),
                                   (290, 287)])
def test_transform_lengths_and_rectangular_grids(kx, ky, mode):
    g = inputs.rng(kx * 1000 + ky)
    pts = g.random((400, 2)) * 2.0 - 0.5
    info = _check(pts, _box_mask(kx, ky, 900, kx + ky), mode=mode, twice=True)
    assert info["n_fine"][0] >= 4 * kx and info["n_fine"][1] >= 4 * ky


@pytest.mark.parametrize("mode", ["kderiv", "direct"])
@pytest.mark.parametrize("K,box", [(2, 1.0), (5, 0.7), (7, 1.0), (13, 2.0)])
def test_transform_lengths_3d(K, box, mode):
    g = inputs.rng(K)
    pts = g.random((500, 3)) * box
    _check(pts, inputs.ball_mask(K, 3), mode=mode, box=box)


@pytest.mark.parametrize("precision", ["f32", "f64"])
@pytest.mark.parametrize("dim,tile", [(2, None), (2, (5, 9)), (2, (9, 5)), (2, (7, 7)), (2, (100, 100)),
                                      (3, None), (3, (8, 6, 5))])
def test_crowded_tiles_bin_again_and_rings_fold(dim, tile, precision):
    """Most points in one clump (the direct form's slots overflow; the compact form bins inside the
    same launch), tiles below, at and above the kernel width, one tile per axis."""
    g = inputs.rng(dim)
    n_bg, n_cl = (9000, 3000) if dim == 2 else (4000, 2500)
    pts = np.vstack([g.random((n_bg, dim)), 0.61 + 0.002 * g.random((n_cl, dim))])
    mask = inputs.ball_mask(14 if dim == 2 else 5, dim)
    _check(pts, mask, precision, width=7 if precision == "f32" else 13, tile=tile, twice=True)


def test_uniform_points_never_leave_the_direct_form_after_an_overflow():
    """An overflow in one call leaves nothing behind for the next."""
    import torch
    from paper_2305_15693_gb300 import fresco
    g = inputs.rng(77)
    mask = inputs.ball_mask(30, 2)
    S0, W = np.zeros(len(mask)), np.ones(len(mask))
    uniform = torch.from_numpy(g.random((20000, 2), dtype=np.float32)).cuda()
    crowded = uniform.clone()
    crowded[:9000] = 0.5 + 0.001 * uniform[:9000]
    with fresco.Plan(1.0, mask, S0, W, 20000, width=7, grad_mode="kderiv") as plan:
        l0, g0 = plan.loss_grad(uniform)
        plan.loss_grad(crowded)
        l1, g1 = plan.loss_grad(uniform)
        torch.cuda.synchronize()
    assert l0.item() == l1.item() and torch.equal(g0, g1)


@pytest.mark.parametrize("shape", [(14, 20), (15, 15), (16, 14), (40, 15), (33, 64), (128, 21)])
def test_half_plane_weights_at_edge_frequencies(shape):
    """Constraints on the folding line (half of the fine grid), at zero, at and beyond the Nyquist
    frequencies, on both signs of the same frequency, on grids around the smallest that run as half
    planes, odd and even."""
    import torch
    from paper_2305_15693_gb300 import fresco
    g = inputs.rng(shape[0] * 100 + shape[1])
    c = g.standard_normal(int(np.prod(shape))).astype(np.float32)
    M = np.array(shape, dtype=np.float64)
    base = (g.random((200, 2)) - 0.5) * 3.0 * M
    edge = np.array([[0.5, 0.5], [-0.5, 0.5], [0.5, 0.0], [0.0, 0.5], [0.0, 0.25], [1.0, 1.0],
                     [0.25, -0.5], [0.5, -0.125]]) * M
    nu = np.vstack([base, edge, -edge[4:], -base[:20]])
    S0, W = 0.2 * g.random(len(nu)), 0.5 + g.random(len(nu))
    want_l, want_g, want_S, _ = oracle.weight_loss_grad_k(
        oracle.grid_points(shape), c.astype(np.float64), 2 * np.pi * nu, S0, W)
    with fresco.Uwnu(shape, nu, S0, W, "f32") as u:
        loss, grad = u.loss_grad(torch.from_numpy(c.reshape(shape[::-1])).cuda())
        l2, _ = u.loss_grad(torch.from_numpy(c.reshape(shape[::-1])).cuda(), want_grad=False)
        S = u.S().double().cpu().numpy()
    assert loss.item() == l2.item()
    assert rel_l2(S, want_S) <= 2e-5
    assert abs(loss.item() - want_l) <= 1e-5 * abs(want_l)
    assert rel_l2(grad.double().cpu().numpy().reshape(-1), want_g) <= 1e-4


@pytest.mark.parametrize("shape,K", [((4, 4), 1), ((64, 22), 9), ((26, 36), 11), ((12, 100), 5),
                                     ((200, 18), 8), ((90, 84), 40), ((2, 2), 0)])
def test_uniform_weights_on_own_and_library_transforms(shape, K):
    """Grids whose lengths factor into the library's radices and grids that keep cuFFT (11, 13), a
    one-sided mask with repeated rows among them; (2, 2) is refused, as its axes are too short."""
    import torch
    from paper_2305_15693_gb300 import fresco
    g = inputs.rng(shape[0] + 7 * shape[1])
    if K == 0:
        with pytest.raises(fresco.FrescoError):
            fresco.Uwu(shape, np.array([[0, 1]], dtype=np.int32), [0.0], [1.0], "f32")
        return
    mask = inputs.ball_mask(K, 2)
    mask = np.vstack([mask[inputs.half_space(mask)], -mask[:3]])
    c = g.standard_normal(int(np.prod(shape))).astype(np.float32)
    S0, W = 0.3 * g.random(len(mask)), 0.2 + g.random(len(mask))
    want_l, want_g, _, _ = oracle.weight_loss_grad(oracle.grid_points(shape), c.astype(np.float64),
                                                   mask, S0, W)
    with fresco.Uwu(shape, mask, S0, W, "f32") as u:
        x = torch.from_numpy(c.reshape(shape[::-1])).cuda()
        l0, _ = u.loss_grad(x, want_grad=False)
        loss, grad = u.loss_grad(x)
        torch.cuda.synchronize()
    assert l0.item() == loss.item()
    assert abs(loss.item() - want_l) <= 1e-5 * abs(want_l)
    assert rel_l2(grad.double().cpu().numpy().reshape(-1), want_g) <= 1e-4
