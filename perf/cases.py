"""Performance cases: what a user of this framework has it evaluate, through its public entry
points, from the smallest problems (launch latency) to the largest that prepare quickly.

Every case is one call a program makes per optimisation step:
  plan      loss and gradient of N points in a periodic box (fresco.Plan, the hot path), 2D or 3D,
            FP32 or FP64, either gradient mode; "autograd" runs it as forward + backward through
            torch.autograd, "pair" adds the hybrid loss's repulsion (fresco.PairTerm)
  lbfgs     a few iterations of the device L-BFGS over such a plan (fresco.LBFGS)
  ensemble  loss and gradient of many independent 2D problems at once (fresco.Batch)
  uwu       real weights on a pixel grid, integer wavevectors (fresco.Uwu)
  uwnu      real weights on a pixel grid, constraints at real frequencies (fresco.Uwnu)
  nuwnu     points with free boundaries, constraints at real wavevectors (fresco.Nuwnu)

The loss of an FP32 plan carries FP32 accuracy in an FP64 scalar; a program that logs it or adds it
to its other FP32 terms takes it as float32, and so do these cases.
"""

import math

import numpy as np
import torch

from paper_2305_15693_gb300 import autograd, fresco

DEV = "cuda"


# ---- cases ---------------------------------------------------------------------------------------

def _plan(name, dim, n, chi, **kw):
    c = {"kind": "plan", "dim": dim, "n": n, "chi": chi, "target": "stealthy", "prec": "f32",
         "mode": "kderiv", "upsample": 2.0, "box": 1.0, "start": "poisson", "via": "loss_grad",
         "pair": False}
    c.update(kw)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest problem: 1024 points, about 630 folded wavevectors, all FP64
        _plan("plan2d_n1024_f64", 2, 1024, 0.3, prec="f64", mode="direct"),
        # a small FP32 problem of a parameter study, odd size, points already optimised (a jittered
        # lattice, some points just outside the box)
        _plan("plan2d_n5003_f32", 2, 5003, 0.4, target="power", start="evolved"),
        # the wrapper's default options (direct gradient mode, oversampling 2) at a common size, on
        # a box that is not the unit one
        _plan("plan2d_n1e5_direct_f32", 2, 100003, 0.3, target="power", mode="direct", box=2.5),
        # 1e6 points, chi = 0.45, stealthy, driven by torch.autograd
        _plan("autograd2d_n1e6_f32", 2, 10**6, 0.45, via="autograd"),
        # the largest 2D problem that prepares quickly: 1e7 points, ten-peak ring target, on the
        # 3-smooth fine grid that needs only w = 7
        _plan("plan2d_n1e7_peaked_f32", 2, 10**7, 0.3, target="peaked", upsample=1.6577),
        # 3D power-law target with the soft-sphere repulsion of the hybrid loss
        _plan("hybrid3d_n2p21_f32", 3, 2**21, 0.3, target="power", upsample=1.6615, pair=True),
        # the accuracy reference in 3D: all FP64, ragged size
        _plan("plan3d_n20011_f64", 3, 20011, 0.25, target="power", prec="f64", mode="direct"),
        # L-BFGS on the smallest problem (ten iterations of its first 200)
        {"name": "lbfgs2d_n1024_f64", "kind": "lbfgs", "n": 1024, "chi": 0.3, "prec": "f64",
         "mode": "direct", "iters": 10},
        # an ensemble of independent configurations, N log-uniform in [1e3, 1e5]
        {"name": "ensemble128_f32", "kind": "ensemble", "n_inst": 128, "n_lo": 1000,
         "n_hi": 100000, "prec": "f32", "mode": "kderiv", "upsample": 1.5, "tile": 64},
        # weights on a pixel grid, integer wavevectors
        {"name": "uwu2d_m1536_f32", "kind": "uwu", "mx": 1536, "my": 1500, "k": 460,
         "prec": "f32"},
        # weights on a 1024^2 grid, 1e6 constraints at real frequencies (a six-fold ring of peaks)
        {"name": "uwnu2d_m1024_k1e6_f32", "kind": "uwnu", "mx": 1024, "my": 1024,
         "n_k": 10**6, "nu_max": 460.0, "prec": "f32"},
        # points with free boundaries and 1e6 real wavevectors (a quasicrystal-like ring of peaks)
        {"name": "nuwnu2d_n1e6_k1e6_f32", "kind": "nuwnu", "n": 10**6, "n_k": 10**6,
         "cycles": 400.0, "prec": "f32"},
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["plan2d", "plan2d", "plan2d", "plan2d_f64", "plan3d", "lbfgs", "ensemble",
                       "uwu", "uwnu", "nuwnu"])
    chi = round(rng.uniform(0.1, 0.5), 3)
    target = rng.choice(["stealthy", "power", "peaked"])
    if kind == "plan2d":
        return _plan(None, 2, _logint(rng, 1000, 4e6), chi, target=target,
                     mode=rng.choice(["kderiv", "kderiv", "direct"]),
                     upsample=rng.choice([2.0, 2.0, 1.65, 1.5]),
                     box=round(rng.uniform(0.5, 3.0), 3),
                     start=rng.choice(["poisson", "evolved"]),
                     via=rng.choice(["loss_grad", "autograd"]))
    if kind == "plan2d_f64":
        return _plan(None, 2, _logint(rng, 500, 2e5), chi, target=target, prec="f64",
                     mode=rng.choice(["kderiv", "direct"]),
                     start=rng.choice(["poisson", "evolved"]))
    if kind == "plan3d":
        f64 = rng.random() < 0.3
        return _plan(None, 3, _logint(rng, 2000, 2e4 if f64 else 1e6), chi, target="power",
                     prec="f64" if f64 else "f32", mode=rng.choice(["kderiv", "kderiv", "direct"]),
                     upsample=rng.choice([2.0, 1.6615]),
                     start=rng.choice(["poisson", "evolved"]), pair=rng.random() < 0.5)
    if kind == "lbfgs":
        f64 = rng.random() < 0.5
        return {"kind": "lbfgs", "n": _logint(rng, 500, 4e3 if f64 else 1e5), "chi": chi,
                "prec": "f64" if f64 else "f32", "mode": rng.choice(["kderiv", "direct"]),
                "iters": rng.choice([3, 4, 5])}
    if kind == "ensemble":
        return {"kind": "ensemble", "n_inst": rng.randint(16, 160), "n_lo": 1000,
                "n_hi": rng.choice([10000, 30000, 100000]), "prec": "f32",
                "mode": rng.choice(["kderiv", "kderiv", "direct"]),
                "upsample": rng.choice([1.5, 2.0]), "tile": rng.choice([0, 32, 48, 64])}
    if kind == "uwu":
        mx, my = _logint(rng, 64, 1536), _logint(rng, 64, 1536)
        return {"kind": "uwu", "mx": mx, "my": my, "prec": rng.choice(["f32", "f32", "f64"]),
                "k": max(4, int(min(mx, my) * rng.uniform(0.1, 0.45)))}
    if kind == "uwnu":
        mx, my = _logint(rng, 64, 1024), _logint(rng, 64, 1024)
        return {"kind": "uwnu", "mx": mx, "my": my, "n_k": _logint(rng, 3000, 1e6),
                "nu_max": round(0.45 * min(mx, my), 1), "prec": "f32"}
    return {"kind": "nuwnu", "n": _logint(rng, 3000, 1e6), "n_k": _logint(rng, 3000, 1e6),
            "cycles": round(rng.uniform(50.0, 400.0), 1), "prec": "f32"}


# ---- inputs --------------------------------------------------------------------------------------

def _dtype(prec):
    return torch.float64 if prec == "f64" else torch.float32


def _gen(seed, stream=0):
    g = torch.Generator(device=DEV)
    g.manual_seed(1000003 * int(seed) + 7919 * stream + 1)
    return g


def _radius(n, dim, chi):
    """Ball radius with about 2 d N chi wavevectors (the constraint ratio chi)."""
    t = 2.0 * dim * n * chi
    return max(2, int(round(math.sqrt(t / math.pi) if dim == 2 else (0.75 * t / math.pi) ** (1 / 3))))


def _ball(k, dim):
    """Every integer n != 0 with |n| <= k: int32 [n_k, dim] on the GPU."""
    r = torch.arange(-k, k + 1, device=DEV, dtype=torch.int32)
    r2 = r.to(torch.int64) ** 2
    s = r2[:, None] + r2[None, :]
    if dim == 3:
        s = s[:, :, None] + r2[None, None, :]
    idx = torch.nonzero((s <= k * k) & (s > 0))
    return (idx - k).to(torch.int32)


def _target(mask, kind, n, k):
    q = mask.double()
    if kind == "power":
        return (q.square().sum(1) / float(k) ** 2)
    s0 = torch.zeros(q.shape[0], device=DEV, dtype=torch.float64)
    if kind == "peaked":
        for p in range(10):
            a = 2.0 * math.pi * p / 10
            d2 = (q[:, 0] - 0.5 * k * math.cos(a)) ** 2 + (q[:, 1] - 0.5 * k * math.sin(a)) ** 2
            s0 += (n / 10.0) * torch.exp(-0.5 * d2)
    return s0


def _points(n, dim, box, start, prec, seed, stream=0):
    g = _gen(seed, stream)
    if start == "poisson":
        x = torch.rand(n, dim, generator=g, device=DEV, dtype=torch.float64)
    else:   # an optimised configuration: a jittered lattice, rows in lattice order
        m = int(math.ceil(n ** (1.0 / dim) - 1e-9))
        i = torch.arange(n, device=DEV)
        x = torch.stack([(i // m ** a) % m for a in range(dim)], 1).double()
        x = (x + 0.7 * torch.rand(n, dim, generator=g, device=DEV, dtype=torch.float64) - 0.35) / m
    return (x * box).to(_dtype(prec)).contiguous()


def _problem(case):
    k = _radius(case["n"], case.get("dim", 2), case["chi"])
    mask = _ball(k, case.get("dim", 2))
    return k, mask, _target(mask, case.get("target", "stealthy"), case["n"], k)


def _ensemble_problem(case, seed):
    """Sizes and masks are the same for every seed (an ensemble's make-up); the points differ."""
    r = np.random.default_rng(7)
    ns = np.rint(np.exp(r.uniform(math.log(case["n_lo"]), math.log(case["n_hi"]),
                                  case["n_inst"]))).astype(int)
    ks = [_radius(int(n), 2, float(c)) for n, c in zip(ns, r.uniform(0.1, 0.5, case["n_inst"]))]
    masks = [_ball(k, 2) for k in ks]
    pts = torch.rand(int(ns.sum()), 2, generator=_gen(seed), device=DEV,
                     dtype=torch.float64).to(_dtype(case["prec"]))
    return [int(n) for n in ns], masks, pts


def _real_k(n_k, kmax, seed, kmin=0.0):
    """Wavevectors uniform in the annulus kmin <= |k| <= kmax, float64 [n_k, 2] on the GPU."""
    u = torch.rand(n_k, 2, generator=_gen(seed, 1), device=DEV, dtype=torch.float64)
    r = torch.sqrt(kmin ** 2 + (kmax ** 2 - kmin ** 2) * u[:, 0])
    a = 2.0 * math.pi * u[:, 1]
    return torch.stack([r * torch.cos(a), r * torch.sin(a)], 1)


def _ring(k, radius, n_peaks, height, width):
    s0 = torch.zeros(k.shape[0], device=DEV, dtype=torch.float64)
    for p in range(n_peaks):
        a = 2.0 * math.pi * p / n_peaks
        d2 = (k[:, 0] - radius * math.cos(a)) ** 2 + (k[:, 1] - radius * math.sin(a)) ** 2
        s0 += height * torch.exp(-0.5 * d2 / width ** 2)
    return s0


def _nuwnu_problem(case, seed):
    x = (torch.rand(case["n"], 2, generator=_gen(seed), device=DEV, dtype=torch.float64) - 0.5)
    kmax = 2.0 * math.pi * case["cycles"]
    # the forward peak of the open box (S ~ N near k = 0) is left unconstrained
    k = _real_k(case["n_k"], kmax, seed, kmin=0.25 * kmax)
    s0 = _ring(k, kmax / (1.0 + math.sqrt(5.0)), 10, 10.0, 2.0 * math.pi)
    return x.to(_dtype(case["prec"])), k, s0


def _weights(case, seed):
    return torch.rand(case["my"], case["mx"], generator=_gen(seed), device=DEV,
                      dtype=torch.float64).to(_dtype(case["prec"]))


def _uwnu_problem(case, seed):
    nu = _real_k(case["n_k"], case["nu_max"], seed)
    return _weights(case, seed), nu, _ring(nu, 0.25 * case["nu_max"], 6, 10.0, 1.0)


def _host(*xs):
    return [x.cpu().numpy() for x in xs]


class State:
    pass


def prepare(case, seed):
    s = State()
    s.kind, s.prec = case["kind"], case["prec"]
    if s.kind in ("plan", "lbfgs"):
        dim, box = case.get("dim", 2), case.get("box", 1.0)
        _, mask, s0 = _problem(case)
        m, t = _host(mask, s0)
        s.plan = fresco.Plan(box, m, t, np.ones(len(t)), case["n"], precision=s.prec,
                             upsample=case.get("upsample", 2.0), grad_mode=case["mode"])
        s.x = _points(case["n"], dim, box, case.get("start", "poisson"), s.prec, seed)
        s.via, s.pair = case.get("via", "loss_grad"), None
        if s.via == "autograd":
            s.x.requires_grad_(True)
        if case.get("pair"):
            s.pair = fresco.PairTerm(box, dim, case["n"],
                                     0.8 * (box ** dim / case["n"]) ** (1.0 / dim),
                                     precision=s.prec)
        if s.kind == "lbfgs":
            s.solver, s.iters = fresco.LBFGS(s.plan), case["iters"]
    elif s.kind == "ensemble":
        ns, masks, s.x = _ensemble_problem(case, seed)
        masks = _host(*masks)
        s.plan = fresco.Batch([1.0] * len(ns), ns, masks, [np.zeros(len(m)) for m in masks],
                              [np.ones(len(m)) for m in masks], precision=s.prec,
                              upsample=case["upsample"], grad_mode=case["mode"],
                              tile=(case["tile"],) * 2 if case["tile"] else None)
    elif s.kind == "uwu":
        m = _ball(case["k"], 2)
        s0 = _target(m, "power", 0, case["k"])
        m, t = _host(m, s0)
        s.plan = fresco.Uwu((case["mx"], case["my"]), m, t, np.ones(len(t)), s.prec)
        s.x = _weights(case, seed)
    elif s.kind == "uwnu":
        s.x, nu, s0 = _uwnu_problem(case, seed)
        nu, s0 = _host(nu, s0)
        s.plan = fresco.Uwnu((case["mx"], case["my"]), nu, s0, np.ones(len(s0)), s.prec)
    else:
        s.x, k, s0 = _nuwnu_problem(case, seed)
        k, s0 = _host(k, s0)
        s.plan = fresco.Nuwnu(1.0, k, s0, np.ones(len(s0)), case["n"], s.prec)
    return s


def run(s):
    if s.kind == "lbfgs":
        x = s.x.clone()
        s.solver.reset()
        rep = s.solver.run(x, s.iters)
        return {"points": x, "loss": rep["loss"]}
    if s.kind == "plan" and s.via == "autograd":
        loss = autograd.structure_factor_loss(s.x, s.plan) / s.x.shape[0]   # loss per point
        grad, = torch.autograd.grad(loss, s.x)
    else:
        loss, grad = s.plan.loss_grad(s.x)
    out = {"loss": loss.detach() if s.prec == "f64" else loss.detach().float(), "grad": grad}
    if s.kind == "plan" and s.pair is not None:
        energy, force = s.pair.energy_grad(s.x.detach())
        out["energy"] = energy if s.prec == "f64" else energy.float()
        out["pair_grad"] = force
    return out


# ---- what one pass cannot do without ----------------------------------------------------------------

def _count(k, dim):
    return math.pi * k * k if dim == 2 else 4.0 / 3.0 * math.pi * k ** 3


def work(case):
    """Points (or weights) read and gradients written once, folded S0 and W per wavevector pair
    read once; the operations of one spread and one interpolation over a 6-cell kernel and of one
    real transform each way at oversampling 1.5."""
    es = 8 if case["prec"] == "f64" else 4

    def transforms(cells):
        return 2.0 * 2.5 * cells * math.log2(max(cells, 2.0))

    def points(n, k, dim):
        n_rep = 0.5 * _count(k, dim)
        return (2.0 * n * dim * es + 2.0 * n_rep * es,
                n * 6.0 ** dim * 6.0 + transforms((3.0 * k) ** dim) + 20.0 * n_rep)

    if case["kind"] in ("plan", "lbfgs"):
        dim = case.get("dim", 2)
        b, f = points(case["n"], _radius(case["n"], dim, case["chi"]), dim)
        if case.get("pair"):
            b += 2.0 * case["n"] * dim * es
            f += case["n"] * 200.0
        if case["kind"] == "lbfgs":
            b, f = b * (case["iters"] + 1), f * (case["iters"] + 1)
    elif case["kind"] == "ensemble":
        r = np.random.default_rng(7)
        ns = np.rint(np.exp(r.uniform(math.log(case["n_lo"]), math.log(case["n_hi"]),
                                      case["n_inst"])))
        b = f = 0.0
        for n, c in zip(ns, r.uniform(0.1, 0.5, case["n_inst"])):
            bi, fi = points(float(n), _radius(int(n), 2, float(c)), 2)
            b, f = b + bi, f + fi
    elif case["kind"] == "uwu":
        cells, n_rep = float(case["mx"] * case["my"]), 0.5 * _count(case["k"], 2)
        b, f = 2.0 * cells * es + 2.0 * n_rep * es, transforms(cells) + 20.0 * n_rep
    else:
        n_k = case["n_k"]
        if case["kind"] == "uwnu":
            n, cells = float(case["mx"] * case["my"]), 2.25 * case["mx"] * case["my"]
            b = 2.0 * n * es
            f = 0.0
        else:
            cells = 2.25 * (3.0 * case["cycles"]) ** 2
            b, f = 4.0 * case["n"] * es, case["n"] * 36.0 * 6.0
        b += n_k * 4.0 * es   # position (2), S0, W
        f += n_k * 36.0 * 8.0 + transforms(cells)
    return {"bytes": b, "flops": f}


# ---- the same in 64 bits: nonuniform transforms in plain torch ---------------------------------------
# Exact to about 1e-13 (2D) and 1e-9 (3D): gridding with a Kaiser-Bessel kernel of width w at
# oversampling 2, FFT in complex128, division by the kernel's closed-form transform.

def _fast_size(n):
    n += n % 2
    while True:
        r = n
        for p in (2, 3, 5, 7):
            while r % p == 0:
                r //= p
        if r == 1:
            return n
        n += 2


class _Gridder:
    """Gridding of points x [N, d] (in cycles of the period, any real value) on a periodic grid of
    nf[a] cells per axis."""

    def __init__(self, x, nf, w):
        self.nf, self.w, self.d = nf, w, x.shape[1]
        self.beta = math.pi * math.sqrt((w / 2.0) ** 2 * 2.25 - 0.8)
        self.i0, self.u, self.wt = [], [], []
        for a in range(self.d):
            t = (x[:, a] - torch.floor(x[:, a])) * nf[a]
            i0 = torch.ceil(t - w / 2.0)
            u = (i0 - t)[:, None] + torch.arange(w, device=x.device, dtype=torch.float64)
            z = torch.sqrt(torch.clamp(1.0 - (2.0 * u / w) ** 2, min=0.0))
            v = torch.special.i0e(self.beta * z) * torch.exp(self.beta * (z - 1.0))
            self.i0.append(i0.long())
            self.u.append(u)
            self.wt.append(v.T.contiguous())

    def ft(self, theta):
        """Transform of the kernel at theta radians per cell (scaled by exp(-beta), as the weights)."""
        s = self.beta ** 2 - (0.5 * self.w * theta) ** 2
        r = torch.sqrt(torch.clamp(s, min=1e-30))
        return self.w * 0.5 * (torch.exp(r - self.beta) - torch.exp(-r - self.beta)) / r

    def cells(self):
        """Every kernel cell of all points: (flat grid index, weight)."""
        def axis(a, k):
            return torch.remainder(self.i0[a] + k, self.nf[a])
        for ky in range(self.w):
            iy, wy = axis(1, ky), self.wt[1][ky]
            for kz in range(self.w if self.d == 3 else 1):
                if self.d == 3:
                    row = (axis(2, kz) * self.nf[1] + iy) * self.nf[0]
                    wr = wy * self.wt[2][kz]
                else:
                    row, wr = iy * self.nf[0], wy
                for kx in range(self.w):
                    yield row + axis(0, kx), wr * self.wt[0][kx]

    def spread(self, c=None):
        """Grids [nf[d-1]..nf[0]] of the point strengths: ones, or each row of c [m, N]."""
        size = int(np.prod(self.nf[:self.d]))
        out = torch.zeros(1 if c is None else c.shape[0], size, device=DEV, dtype=torch.float64)
        for i, v in self.cells():
            if c is None:
                out[0].index_add_(0, i, v)
            else:
                for q in range(c.shape[0]):
                    out[q].index_add_(0, i, v * c[q])
        return out.reshape((-1,) + tuple(self.nf[a] for a in range(self.d - 1, -1, -1)))

    def interp(self, grids):
        """Values [m, N] of real grids [m, ...] at the points."""
        g = grids.reshape(grids.shape[0], -1)
        out = torch.zeros(g.shape[0], self.i0[0].shape[0], device=DEV, dtype=torch.float64)
        for i, v in self.cells():
            for q in range(g.shape[0]):
                out[q] += g[q][i] * v
        return out


def _psi(gr, a, n):
    return gr.ft(2.0 * math.pi * n.double() / gr.nf[a])


def _index(gr, n):
    """Flat grid index of integer frequencies n [n_k, d]."""
    i = torch.remainder(n[:, gr.d - 1].long(), gr.nf[gr.d - 1])
    for a in range(gr.d - 2, -1, -1):
        i = i * gr.nf[a] + torch.remainder(n[:, a].long(), gr.nf[a])
    return i


def _modes(gr, n):
    """Product of the kernel's transforms at integer frequencies n."""
    p = 1.0
    for a in range(gr.d):
        p = p * _psi(gr, a, n[:, a])
    return p


def _exact_points(x, box, mask, s0, k, w):
    """(loss, gradient) of the points x for the ball mask and targets, W = 1."""
    n, d = x.shape
    gr = _Gridder(x.double() / box, [_fast_size(max(2 * (2 * k + 1), 2 * w))] * d, w)
    shape = tuple(gr.nf[:d])
    psi, idx = _modes(gr, mask), _index(gr, mask)
    rho = torch.fft.fftn(gr.spread()[0].to(torch.complex128)).reshape(-1)[idx] / psi
    dev = (rho.real ** 2 + rho.imag ** 2) / n - s0
    e = 4.0 * dev * rho / n / psi
    fields = []
    for a in range(d):
        f = torch.zeros(shape, device=DEV, dtype=torch.complex128).reshape(-1)
        f[idx] = 1j * (2.0 * math.pi / box) * mask[:, a].double() * e
        f = torch.fft.ifftn(f.reshape(shape), norm="forward")
        fields.append(f.real.contiguous())
    return (dev ** 2).sum(), gr.interp(torch.stack(fields)).T.contiguous()


def _exact_pair(x, box, sigma, cap=24):
    """(energy, gradient) of the harmonic soft spheres (1 - r / sigma)^2 / 2, r < sigma."""
    n, d = x.shape
    x = x.double()
    x = x - box * torch.floor(x / box)
    m = max(1, int(math.floor(box / sigma)))
    if m < 3 or n > 4_000_000:
        return None, None
    c = torch.clamp((x * (m / box)).long(), max=m - 1)
    lin = c[:, 0]
    for a in range(1, d):
        lin = lin + c[:, a] * m ** a
    order = torch.argsort(lin)
    first = torch.searchsorted(lin[order], torch.arange(m ** d, device=DEV))
    rank = torch.empty_like(lin)
    rank[order] = torch.arange(n, device=DEV) - first[lin[order]]
    if int(rank.max()) >= cap:
        return None, None
    table = torch.full((m ** d, int(rank.max()) + 1), -1, device=DEV, dtype=torch.long)
    table[lin, rank] = torch.arange(n, device=DEV)
    energy = torch.zeros((), device=DEV, dtype=torch.float64)
    grad = torch.zeros_like(x)
    for o in range(3 ** d):
        nb = torch.zeros_like(lin)
        for a in range(d):
            nb += torch.remainder(c[:, a] + (o // 3 ** a) % 3 - 1, m) * m ** a
        for q in range(table.shape[1]):
            j = table[nb, q]
            ok = (j >= 0) & (j != torch.arange(n, device=DEV))
            v = x - x[torch.clamp(j, min=0)]
            v = v - box * torch.round(v / box)
            r = torch.sqrt((v * v).sum(1))
            ok = ok & (r < sigma) & (r > 0)
            u = torch.where(ok, 1.0 - r / sigma, torch.zeros_like(r))
            energy += 0.25 * (u * u).sum()
            grad -= torch.where(ok, u / (sigma * r), torch.zeros_like(r))[:, None] * v
    return energy, grad


def _exact_at(c, ix, nu, s0, scale, norm, w):
    """Sums over the nonzero grid weights c [my, mx] at signed integer positions ix = (x, y) for
    real frequencies nu (cycles per grid length m = c's extents), with a factor `scale` per
    frequency: returns (S, deviation, type-1 sum G on the grid)."""
    my, mx = c.shape
    x = -nu / torch.tensor([mx, my], device=DEV, dtype=torch.float64)
    gr = _Gridder(x, [_fast_size(max(2 * mx, 2 * w)), _fast_size(max(2 * my, 2 * w))], w)
    sx, sy = ix
    psi = _psi(gr, 1, sy)[:, None] * _psi(gr, 0, sx)[None, :]
    at = (torch.remainder(sy, gr.nf[1])[:, None], torch.remainder(sx, gr.nf[0])[None, :])
    u = torch.zeros(gr.nf[1], gr.nf[0], device=DEV, dtype=torch.complex128)
    u[at] = (c / psi).to(torch.complex128)
    u = torch.fft.ifft2(u, norm="forward")
    rho = gr.interp(torch.stack([u.real.contiguous(), u.imag.contiguous()])) * scale
    s = (rho ** 2).sum(0) / norm
    dev = s - s0
    coef = 4.0 * dev * rho * scale / norm
    t = gr.spread(coef)
    g = torch.fft.fft2(torch.complex(t[0], t[1]))[at].real / psi
    return s, dev, g


def _signed(m, half_up):
    """Signed positions of m cells: centred (pixel grids) or wrapped past the middle."""
    i = torch.arange(m, device=DEV)
    return i - m // 2 if half_up else torch.where(i < m // 2, i, i - m)


def exact(case, seed):
    kind = case["kind"]
    if kind == "lbfgs":
        return None
    if kind == "plan":
        dim, box = case["dim"], case["box"]
        k, mask, s0 = _problem(case)
        x = _points(case["n"], dim, box, case["start"], case["prec"], seed)
        w = 16 if dim == 2 or case["prec"] == "f64" else 10
        loss, grad = _exact_points(x, box, mask, s0, k, w)
        if case["via"] == "autograd":
            loss, grad = loss / case["n"], grad / case["n"]
        out = {"loss": loss, "grad": grad}
        if case["pair"]:
            sigma = 0.8 * (box ** dim / case["n"]) ** (1.0 / dim)
            out["energy"], out["pair_grad"] = _exact_pair(x, box, sigma)
        return out
    if kind == "ensemble":
        ns, masks, pts = _ensemble_problem(case, seed)
        loss, grad, first = [], [], 0
        for n, m in zip(ns, masks):
            k = int(m.max())
            le, ge = _exact_points(pts[first:first + n], 1.0, m, torch.zeros(len(m), device=DEV),
                                   k, 12)
            loss.append(le)
            grad.append(ge)
            first += n
        return {"loss": torch.stack(loss), "grad": torch.cat(grad)}
    if kind == "uwu":
        c = _weights(case, seed).double()
        m = _ball(case["k"], 2).long()
        s0 = _target(m, "power", 0, case["k"])
        rho = torch.fft.fft2(c.to(torch.complex128))
        at = (torch.remainder(m[:, 1], case["my"]), torch.remainder(m[:, 0], case["mx"]))
        norm = (c * c).sum()
        s = (rho[at].real ** 2 + rho[at].imag ** 2) / norm
        e = torch.zeros_like(rho)
        e[at] = 4.0 * (s - s0) * rho[at] / norm
        grad = torch.fft.ifft2(e, norm="forward").real - 4.0 * c / norm * (s * (s - s0)).sum()
        return {"loss": ((s - s0) ** 2).sum(), "grad": grad}
    if kind == "uwnu":
        c, nu, s0 = _uwnu_problem(case, seed)
        c = c.double()
        norm = (c * c).sum()
        s, dev, g = _exact_at(c, (_signed(case["mx"], True), _signed(case["my"], True)), nu, s0,
                              1.0, norm, 16)
        return {"loss": (dev ** 2).sum(), "grad": g - 4.0 * c / norm * (s * dev).sum()}
    # nuwnu: the points on an oversampled grid of spacing h, then as weights on that grid
    x, k, s0 = _nuwnu_problem(case, seed)
    w = 16
    kmax = 2.0 * math.pi * case["cycles"]
    h = math.pi / (2.0 * kmax)
    m = _fast_size(int(math.ceil(1.0 / h)) + w + 2)
    gr = _Gridder(x.double() / (m * h), [m, m], w)
    b = gr.spread()[0]
    theta = k * h
    scale = 1.0 / (gr.ft(theta[:, 0]) * gr.ft(theta[:, 1]))
    ix = (_signed(m, False), _signed(m, False))
    _, dev, g = _exact_at(b, ix, theta * m / (2.0 * math.pi), s0, scale, float(case["n"]), w)
    grad = _gradient_of_interpolant(gr, g, h)
    return {"loss": (dev ** 2).sum(), "grad": grad}


def _gradient_of_interpolant(gr, g, h):
    """d/dr of sum_l g_l psi(l - r / h) at the points: the kernel's derivative along each axis."""
    out = []
    for a in range(2):
        keep = gr.wt[a]
        t = gr.u[a]
        z = torch.sqrt(torch.clamp(1.0 - (2.0 * t / gr.w) ** 2, min=1e-300))
        dz = -(4.0 * t / gr.w ** 2) / z
        gr.wt[a] = (gr.beta * dz * torch.special.i1e(gr.beta * z)
                    * torch.exp(gr.beta * (z - 1.0))).T.contiguous()
        out.append(-gr.interp(g[None])[0] / h)
        gr.wt[a] = keep
    return torch.stack(out, 1)
