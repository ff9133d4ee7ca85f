"""The tests of the NUFFT path whose problems are small enough that a plan with default options runs
them as direct sums, run again on plans that name their tiles (the ones the options would choose, so
that grid and kernel width stay what they were), so that binning, tiles, spread, transforms and
interpolation are what they exercise: the parity tests, the FP64 tiles at every width, and the
tile-ordered solver. Every evaluation asserts that it was not the direct sums' two or three
launches."""

import inspect
import itertools

import pytest

import test_gpu_f64_tiles as tiles
import test_gpu_optim as optim
import test_gpu_parity as parity

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import torch
    from paper_2305_15693_gb300 import _build
    assert torch.cuda.is_available(), "GPU tests need CUDA"
    _build.build()


def _calls(fn):
    """Every argument set of a parametrised test function, as (id, keyword arguments)."""
    axes = []
    for mark in getattr(fn, "pytestmark", []):
        if mark.name == "parametrize":
            names = [n.strip() for n in mark.args[0].split(",")]
            axes.append([dict(zip(names, v if len(names) > 1 else (v,))) for v in mark.args[1]])
    for parts in itertools.product(*axes):
        kw = {k: v for p in parts for k, v in p.items()}
        yield "-".join([fn.__name__[5:]] + [str(v) for v in kw.values() if not isinstance(v, dict)]), kw


def _tests(module, *names):
    fns = [f for n, f in vars(module).items()
           if n.startswith("test_") and inspect.isfunction(f) and (not names or n in names)]
    return [pytest.param(f, kw, id=i) for f in fns for i, kw in _calls(f)]


CASES = (_tests(parity) + _tests(tiles) +
         _tests(optim, "test_tile_ordered_solver_follows_the_reference_and_returns_caller_order"))


@pytest.mark.parametrize("test,args", CASES)
def test_on_the_nufft(test, args, monkeypatch):
    from paper_2305_15693_gb300 import fresco

    class NufftPlan(fresco.Plan):
        def __init__(self, box, mask, S0, W, n_points, **kw):
            q = None
            if not kw.get("width") and not kw.get("tile"):
                o = {k: v for k, v in kw.items() if k != "stream"}
                q = fresco.fresco_plan_query(box, mask, S0, W, n_points, fresco.make_opts(**o))
                kw["tile"] = q["tile"]
            super().__init__(box, mask, S0, W, n_points, **kw)
            same = ("n_fine", "width", "beta")
            assert q is None or all(q[k] == self.info[k] for k in same)

        def _counted(self, call, *a, **kw):
            n = self.launch_count()
            out = call(*a, **kw)
            assert self.launch_count() - n > 3
            return out

        def loss_grad(self, *a, **kw):
            return self._counted(super().loss_grad, *a, **kw)

        def forward(self, *a, **kw):
            return self._counted(super().forward, *a, **kw)

    monkeypatch.setattr(fresco, "Plan", NufftPlan)
    test(**args)
