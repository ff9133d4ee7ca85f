"""The pair term's energy is summed as exactly as in FP64 in both precisions (the terms are those of
the plan's precision): sums beyond FP32's range stay finite and right, and terms that are infinite
make the energy infinite."""

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


@pytest.mark.parametrize("dim,sigma", [(2, 0.2), (3, 0.2), (2, 0.45)])
def test_energy_beyond_the_range_of_fp32(dim, sigma):
    """120 points close together: every pair's energy is within FP32's range and one point's sum over
    its pairs is not. (sigma = 0.45: the form for fewer than three cells an axis.) Each FP32 term is
    within a few ulp: 1e-5 relative."""
    import torch
    from paper_2305_15693_gb300 import fresco
    n, eps = 120, 3e37
    x = (0.3 + 0.02 * inputs.rng(dim).random((n, dim))).astype(np.float32)
    d = x.astype(np.float64)[:, None] - x.astype(np.float64)[None]
    r = np.sqrt((d ** 2).sum(-1))[np.triu_indices(n, 1)]
    want = np.sum(eps / 2.0 * (1.0 - r / sigma) ** 2)
    p = fresco.PairTerm(1.0, dim, n, sigma, eps, 2.0, "f32")
    energy, _ = p.energy_grad(torch.from_numpy(x).cuda())
    torch.cuda.synchronize()
    p.close()
    assert abs(energy.item() - want) <= 1e-5 * want


def _energy(x, dim, sigma, eps, box=1.0):
    import torch
    from paper_2305_15693_gb300 import fresco
    p = fresco.PairTerm(box, dim, len(x), sigma, eps, 2.0, "f32")
    energy, _ = p.energy_grad(torch.from_numpy(x).cuda())
    torch.cuda.synchronize()
    p.close()
    return energy.item()


def test_infinite_terms_give_an_infinite_energy():
    """eps / alpha overflows FP32 (every term is infinite), as it would in a sum in FP64."""
    x = (0.3 + 0.02 * inputs.rng(3).random((50, 2))).astype(np.float32)
    assert _energy(x, 2, 0.2, 1e39) == np.inf
