"""Pairs whose distance is the potential's range to the last bit: r^2 < sigma^2 as rounded while r /
sigma rounds to more than 1. Their energy and force are zero, not the square root or power of a negative
number."""

from fractions import Fraction

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    from paper_2305_15693_gb300 import _build
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    _build.build()


def _edge(dt, lo, hi):
    """sigma and a separation (a, b) of type dt whose squared distance, as the kernel rounds it (a a, then
    fma(b, b, .)), is below sigma^2 and whose square root times 1 / sigma is beyond 1."""
    g = np.random.default_rng(5)
    for _ in range(20000):
        sigma = dt(g.uniform(lo, hi))
        inv, sig2 = dt(1) / sigma, sigma * sigma
        if Fraction(float(sigma)) * Fraction(float(inv)) <= 1:
            continue
        b = dt(g.uniform(0.1, 0.9)) * sigma
        a = np.sqrt(sig2 - b * b)
        r2 = dt(Fraction(float(b)) ** 2 + Fraction(float(a * a)))   # (correctly rounded in FP64)
        if r2 < sig2 and Fraction(float(np.sqrt(r2))) * Fraction(float(inv)) > 1:
            return sigma, a, b
    raise AssertionError("no such pair found")


@pytest.mark.parametrize("alpha", [2.0, 2.5, 1.7, 3.2])
@pytest.mark.parametrize("lo,hi", [(0.1, 0.2), (0.36, 0.45)])
@pytest.mark.parametrize("dim,precision", [(2, "f32"), (3, "f32"), (2, "f64"), (3, "f64")])
def test_pairs_at_the_cutoff(dim, precision, lo, hi, alpha):
    import torch
    from paper_2305_15693_gb300 import fresco
    dt = np.float64 if precision == "f64" else np.float32
    sigma, a, b = _edge(dt, lo, hi)
    x = np.zeros((2, dim), dtype=dt)
    x[1, 0], x[1, 1] = a, b
    p = fresco.PairTerm(1.0, dim, 2, float(sigma), 1.0, alpha, precision)
    energy, grad = p.energy_grad(torch.from_numpy(x).cuda())
    torch.cuda.synchronize()
    p.close()
    eps = float(np.finfo(dt).eps)
    assert abs(energy.item()) <= 4 * eps
    assert np.all(np.abs(grad.cpu().numpy()) <= (4 * eps) ** min(1.0, alpha - 1.0) * 10)
