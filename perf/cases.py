"""The work that users of this library have it do, as cases that can be timed and compared.

A case is one call (or one round of requests) through the public entry points of
``paper_1505_02248_gb300.lem``: ``Lem.step``, ``Lem.build``, ``Batch.run`` and ``Server``. The
problems are the repository's own model problems (heat, advection-diffusion, variable diffusion
with a reaction, Schroedinger, porous medium) at its own sizes and at odd ones between them.

``exact`` steps the same problems in 64 bits with torch alone: window by window, the local
exponential acts through a scaled Taylor series of the stencil (or, where all windows share one
operator, through one dense matrix made by scaling and doubling).
"""
import math

import numpy as np
import torch

from paper_1505_02248_gb300 import lem

DEV = "cuda"
F64 = torch.float64


# --------------------------------------------------------------------------- the cases
def listed():
    return [
        # A small 1D problem stepped in short calls: launches and latency are everything.
        dict(name="heat1d_1024_fp64", kind="heat1d", n=1024, tile=64, overlap=16, mu=10.0, prec="fp64", steps=10),
        # The headline: a large periodic 2D field on the mixed-precision tier.
        dict(name="advdiff2d_2048_split", kind="advdiff2d", side=2048, tile=32, overlap=8, mu=20.0, cx=4.0,
             prec="split", steps=10),
        # The two-piece tier on a mid-sized field with a tile that is no power of two.
        dict(name="advdiff2d_648_split_fast", kind="advdiff2d", side=648, tile=24, overlap=7, mu=12.0, cx=2.0,
             prec="split_fast", steps=10),
        # The FP64 tier, the library's precise answer and the server's 1e-10 tier.
        dict(name="advdiff2d_1024_fp64", kind="advdiff2d", side=1024, tile=32, overlap=8, mu=20.0, cx=4.0,
             prec="fp64", steps=4),
        # FP64 between walls, odd mesh, tiles that do not divide it, the exponential mode: many small
        # classes of windows beside one large one.
        dict(name="walls2d_389x517_exp_fp64", kind="walls2d", ny=389, nx=517, ty=24, tx=32, oy=6, ox=8, mu=8.0,
             mode="exp", prec="fp64", steps=4),
        # Variable coefficients with the reaction, a propagator for every tile, FP32 storage.
        dict(name="vardiff2d_320_split_fast", kind="vardiff2d", side=320, tile=16, overlap=6, prec="split_fast",
             refresh=0, steps=10),
        # The same problem kind with its Jacobian refreshed every step: each step builds propagators.
        dict(name="vardiff2d_80_refresh_split", kind="vardiff2d", side=80, tile=16, overlap=6, prec="split",
             refresh=1, steps=2),
        # A long 1D line of variable diffusion with truncated propagators.
        dict(name="vardiff1d_300001_trunc", kind="vardiff1d", n=300001, tile=64, overlap=16, tol=1e-8,
             prec="split_fast", steps=10),
        # Complex states: a Schroedinger line.
        dict(name="schrodinger1d_65536_split_fast", kind="schrodinger1d", n=65536, tile=80, overlap=20, mu=2.0,
             prec="split_fast", steps=10),
        # The porous medium, Jacobian refreshed every step in FP64: small builds, one after another.
        dict(name="porous1d_400_refresh_fp64", kind="porous1d", n=400, tile=40, overlap=12, mu=4.0, refresh=1,
             prec="fp64", steps=4),
        # Uneven problems advanced together by one graph launch.
        dict(name="batch_24_uneven_split", kind="batch", count=24, side_max=512, pick=3, prec="split", steps=10),
        # A round of requests to a server that already holds their operators: both tolerance tiers,
        # 1D and 2D, host states in and out.
        dict(name="serve_12_mixed", kind="serve", count=12, pick=5),
    ]


def _logint(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the listed kinds, its sizes spread over what the listed ones span."""
    kind = rng.choice(["heat1d", "advdiff2d", "advdiff2d", "advdiff64", "walls2d", "vardiff2d", "refresh2d",
                       "vardiff1d", "schrodinger1d", "porous1d", "batch", "serve"])
    if kind == "heat1d":
        tile = rng.choice([16, 32, 50, 64])
        return dict(kind=kind, n=_logint(rng, 256, 16384), tile=tile, overlap=rng.randint(4, 20),
                    mu=round(rng.uniform(1, 20), 3), prec="fp64", steps=rng.choice([1, 4, 10, 50]))
    if kind == "advdiff2d":
        tile = rng.choice([8, 16, 24, 32])
        side = tile * max(2, _logint(rng, 128, 1600) // tile)
        return dict(kind=kind, side=side, tile=tile, overlap=rng.randint(4, 8), mu=round(rng.uniform(1, 50), 3),
                    cx=round(rng.uniform(0, 4), 3), prec=rng.choice(["split", "split_fast"]),
                    steps=rng.choice([1, 4, 10]))
    if kind == "advdiff64":
        tile = rng.choice([8, 13, 16, 24, 32])
        side = tile * max(2, _logint(rng, 64, 900) // tile)
        return dict(kind="advdiff2d", side=side, tile=tile, overlap=rng.randint(3, 8), mu=round(rng.uniform(1, 50), 3),
                    cx=round(rng.uniform(0, 4), 3), prec="fp64", steps=rng.choice([1, 2, 4]))
    if kind == "walls2d":
        return dict(kind=kind, ny=_logint(rng, 60, 600), nx=_logint(rng, 60, 600), ty=rng.randint(8, 32),
                    tx=rng.randint(8, 32), oy=rng.randint(2, 8), ox=rng.randint(2, 8), mu=round(rng.uniform(1, 20), 3),
                    mode=rng.choice(["phi", "exp"]), prec="fp64", steps=rng.choice([1, 4]))
    if kind == "vardiff2d":
        tile, overlap = rng.choice([(8, 3), (8, 4), (12, 4), (16, 5), (16, 6)])
        prec = rng.choice(["split_fast", "split_fast", "split"])
        return dict(kind=kind, side=_logint(rng, 64, 320), tile=tile, overlap=overlap, prec=prec, refresh=0,
                    steps=rng.choice([2, 10]))
    if kind == "refresh2d":
        tile, overlap = rng.choice([(8, 3), (8, 4), (12, 4), (16, 6)])
        return dict(kind="vardiff2d", side=_logint(rng, 32, 80), tile=tile, overlap=overlap, prec="split",
                    refresh=1, steps=2)
    if kind == "vardiff1d":
        return dict(kind=kind, n=_logint(rng, 5000, 400000), tile=rng.choice([32, 64, 96]), overlap=rng.randint(8, 24),
                    tol=rng.choice([1e-8, 1e-10]), prec=rng.choice(["split_fast", "fp64"]), steps=rng.choice([2, 10]))
    if kind == "schrodinger1d":
        return dict(kind=kind, n=_logint(rng, 400, 65536), tile=rng.choice([40, 64, 80]), overlap=rng.randint(10, 24),
                    mu=round(rng.uniform(1, 4), 3), prec=rng.choice(["split_fast", "fp64"]), steps=rng.choice([2, 10]))
    if kind == "porous1d":
        return dict(kind=kind, n=_logint(rng, 100, 2000), tile=rng.choice([20, 40, 50]), overlap=rng.randint(6, 16),
                    mu=round(rng.uniform(1, 6), 3), refresh=1, prec="fp64", steps=rng.choice([2, 4]))
    if kind == "batch":
        return dict(kind=kind, count=rng.randint(3, 24), side_max=rng.choice([128, 256, 512]),
                    pick=rng.randint(10, 10 ** 6), prec="split", steps=rng.choice([4, 10]))
    return dict(kind="serve", count=rng.randint(4, 12), pick=rng.randint(10, 10 ** 6))


# --------------------------------------------------------------------------- problems and fields
def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    return g


def _field(shape, ell, g):
    """A Gaussian random field of correlation length ell nodes, zero mean, unit deviation."""
    w = torch.randn(shape, generator=g, device=DEV, dtype=F64)
    ks = [2 * math.pi * torch.fft.fftfreq(n, device=DEV, dtype=F64) for n in shape]
    k2 = sum((k.reshape([-1 if a == b else 1 for b in range(len(shape))])) ** 2 for a, k in enumerate(ks))
    f = torch.fft.ifftn(torch.fft.fftn(w) * torch.exp(-k2 * ell ** 2 / 4)).real
    f = f - f.mean()
    return (f / f.std()).contiguous()


def _walled_field(shape, ell, g):
    """The same, not periodic: a corner of a larger one."""
    f = _field(tuple(2 * n for n in shape), ell, g)
    for a, n in enumerate(shape):
        f = f.narrow(a, 0, n)
    f = f - f.mean()
    return (f / f.std()).contiguous()


def _upwind2d(mu, cx, cy):
    """-(cx, cy) . grad u + mu Laplacian u on unit spacing, first-order upwind."""
    return {"C": -4 * mu - cx - cy, "W": mu + cx, "E": mu, "S": mu + cy, "N": mu}


def _faces(k, h):
    """div(k grad u): face values are means of the two nodes', at a wall the node's own."""
    co = {"C": 0.0}
    for axis, (lo, hi) in enumerate((("S", "N"), ("W", "E")) if k.dim() == 2 else (("W", "E"),)):
        n = k.shape[axis]
        first, last = k.narrow(axis, 0, 1), k.narrow(axis, n - 1, 1)
        mid = (k.narrow(axis, 1, n - 1) + k.narrow(axis, 0, n - 1)) / 2
        co[lo] = torch.cat([first, mid], axis) / h ** 2
        co[hi] = torch.cat([mid, last], axis) / h ** 2
        co["C"] = co["C"] - co[lo] - co[hi]
    return co


class Problem:
    """What a user states: mesh, walls, stencil, step, tiles, and an initial field."""

    def __init__(self, shape, bc, coef, dt, tile, overlap, u0, mode="phi", reaction=False, refresh=0, porous_m=0.0):
        self.shape, self.bc, self.coef, self.dt = tuple(shape), bc, coef, float(dt)
        self.tile, self.overlap, self.u0, self.mode = tuple(tile), tuple(overlap), u0, mode
        self.reaction, self.refresh, self.porous_m = reaction, refresh, porous_m

    def arrays(self):
        return {k: v.cpu().numpy().ravel() if isinstance(v, torch.Tensor) else v for k, v in self.coef.items()}

    def context(self, prec):
        return lem.Lem(self.shape, self.bc, self.arrays(), self.dt, self.tile, self.overlap, mode=self.mode, prec=prec,
                       reaction=self.reaction, refresh=self.refresh, porous_m=self.porous_m)


def _advdiff(side, tile, overlap, mu, cx, u0):
    return Problem((side, side), ("periodic",) * 2, _upwind2d(mu, cx, cx / 2), 1.0, (tile,) * 2, (overlap,) * 2, u0)


def _heat1d(n, tile, overlap, mu, u0):
    return Problem((n,), ("dirichlet",), {"C": -2.0 * mu, "W": mu, "E": mu}, 1.0, (tile,), (overlap,), u0)


def _sines(n, g):
    """Eight sine modes with normal amplitudes: what a heated rod starts from."""
    a = torch.randn(8, generator=g, device=DEV, dtype=F64)
    j = torch.arange(1, n + 1, device=DEV, dtype=F64)
    k = torch.arange(1, 9, device=DEV, dtype=F64)
    return (a[:, None] * torch.sin(math.pi * k[:, None] * j / (n + 1))).sum(0).contiguous()


def _problem(case, seed):
    g = _gen(seed)
    kind = case["kind"]
    if kind == "heat1d":
        return _heat1d(case["n"], case["tile"], case["overlap"], case["mu"], _sines(case["n"], g))
    if kind == "advdiff2d":
        side = case["side"]
        return _advdiff(side, case["tile"], case["overlap"], case["mu"], case["cx"], _field((side, side), 16.0, g))
    if kind == "walls2d":
        shape = (case["ny"], case["nx"])
        return Problem(shape, ("dirichlet",) * 2, _upwind2d(case["mu"], 1.0, 0.5), 1.0, (case["ty"], case["tx"]),
                       (case["oy"], case["ox"]), _walled_field(shape, 12.0, g), mode=case["mode"])
    if kind == "vardiff2d":
        side = case["side"]
        k = torch.exp(_walled_field((side, side), 32.0, g))
        u0 = 0.5 * _walled_field((side, side), 16.0, g)
        h = 1.0 / (side + 1)
        return Problem((side, side), ("dirichlet",) * 2, _faces(k, h), 2.0 * h * h / float(k.median()),
                       (case["tile"],) * 2, (case["overlap"],) * 2, u0, reaction=True, refresh=case["refresh"])
    if kind == "vardiff1d":
        n = case["n"]
        k = torch.exp(_walled_field((n,), 32.0, g))
        h = 1.0 / (n + 1)
        return Problem((n,), ("dirichlet",), _faces(k, h), 2.0 * h * h / float(k.median()), (case["tile"],),
                       (case["overlap"],), _walled_field((n,), 16.0, g))
    if kind == "schrodinger1d":
        # (i/2) c_xx - i (kappa/2) x^2 c, a ring of n nodes; a packet of smooth random waves
        n, length, kappa = case["n"], 10.0, 10.0
        h = length / n
        x = -length / 2 + h * torch.arange(n, device=DEV, dtype=F64)
        u0 = torch.complex(_field((n,), 16.0, g), _field((n,), 16.0, g)) * torch.exp(-x * x / 8)
        one = torch.ones_like(x)
        coef = {"C": torch.complex(0 * x, -one / h ** 2 - kappa * x * x / 2), "W": torch.complex(0 * x, one / (2 * h * h)),
                "E": torch.complex(0 * x, one / (2 * h * h))}
        return Problem((n,), ("periodic",), coef, 2 * case["mu"] * h * h, (case["tile"],), (case["overlap"],), u0)
    if kind == "porous1d":
        # c_t = (c^3)_xx from a Barenblatt bump whose size the seed sets
        n, length, m = case["n"], 10.0, 3.0
        h = length / (n + 1)
        x = -length / 2 + h * (torch.arange(n, device=DEV, dtype=F64) + 1)
        amp = 0.8 + 0.4 * float(torch.rand(1, generator=g, device=DEV, dtype=F64))
        k = 1 / (m + 1)
        u0 = torch.clamp(amp * amp - k * (m - 1) * x * x / (2 * m), min=0) ** (1 / (m - 1))
        dt = case["mu"] * h * h / (m * float(u0.max()) ** (m - 1))
        return Problem((n,), ("dirichlet",), {"C": -2 / h ** 2, "W": 1 / h ** 2, "E": 1 / h ** 2}, dt, (case["tile"],),
                       (case["overlap"],), u0.contiguous(), refresh=case["refresh"], porous_m=m)
    raise ValueError(kind)


def _batch(case, seed):
    """Independent periodic problems of uneven size (the pick sets them, the seed their fields)."""
    r, g, out = np.random.RandomState(case["pick"] % (1 << 31)), _gen(seed), []
    for _ in range(case["count"]):
        side = 32 * r.randint(2, case["side_max"] // 32 + 1)
        tile, overlap = int(r.choice([8, 16, 32])), r.randint(4, 9)
        mu, cx = r.uniform(1, 50), r.uniform(0, 4)
        out.append(_advdiff(int(side), tile, int(overlap), float(mu), float(cx), _field((side, side), 8.0, g)))
    return out


def _requests(case, seed):
    """(problem, tolerance, steps) of one round of requests; a user base shares a few operators."""
    r, g, out = np.random.RandomState(case["pick"] % (1 << 31)), _gen(seed), []
    for q in range(case["count"]):
        steps, tol = int(r.randint(1, 21)), 1e-10 if q % 3 == 2 else 1e-6
        if q % 4 == 3:
            n = int(round(math.exp(r.uniform(math.log(256), math.log(65536)))))
            out.append((_heat1d(n, 64, 16, 10.0, _sines(n, g)), tol, steps))
        else:
            side = 32 * int(r.randint(4, 17 if tol > 1e-8 else 9))
            mu, cx = ((5.0, 1.0), (20.0, 4.0))[q % 2]
            out.append((_advdiff(side, (16, 32)[q % 2], (6, 8)[q % 2], mu, cx, _field((side, side), 12.0, g)), tol, steps))
    return out


# --------------------------------------------------------------------------- prepare and run
def prepare(case, seed):
    if case["kind"] == "batch":
        probs = _batch(case, seed)
        ctxs = [p.context(case["prec"]) for p in probs]
        u0 = torch.cat([p.u0.reshape(-1) for p in probs])
        u = u0.clone()
        states = list(torch.split(u, [p.u0.numel() for p in probs]))
        return dict(kind="batch", ctxs=ctxs, u0=u0, u=u, states=states,
                    batch=lem.Batch(ctxs, states, steps_per_launch=case["steps"]))
    if case["kind"] == "serve":
        reqs = [(p.shape, p.bc, p.arrays(), p.dt, p.tile, p.overlap, p.u0.cpu().numpy().ravel().copy(), steps, tol)
                for p, tol, steps in _requests(case, seed)]
        st = dict(kind="serve", server=lem.Server(), requests=reqs, bufs=[np.empty_like(q[6]) for q in reqs])
        run(st)  # the server in use holds its operators already
        return st
    p = _problem(case, seed)
    ctx = p.context(case["prec"])
    if case.get("tol") is not None:
        ctx.set_truncation(case["tol"])
    u0 = p.u0.reshape(-1).contiguous()
    if not case.get("refresh"):
        ctx.build(u0 if p.reaction else None)
        if case.get("tol") is not None:
            ctx.band_total()
    return dict(kind="step", ctx=ctx, u0=u0, steps=case["steps"], refresh=case.get("refresh", 0))


def run(st):
    """One pass: a new field advanced by the case's steps (or a round of fields)."""
    if st["kind"] == "batch":
        st["u"].copy_(st["u0"])
        st["batch"].run(1)
        return st["states"]
    if st["kind"] == "serve":
        srv, tickets = st["server"], []
        for q, buf in zip(st["requests"], st["bufs"]):
            np.copyto(buf, q[6])
            tickets.append(srv.submit(*q[:6], buf, q[7], tol=q[8]))
        for t in tickets:
            srv.wait(t)
        return st["bufs"]
    u = st["u0"].clone()
    if st["refresh"]:
        st["ctx"].build(u)  # a new field's first Jacobian
    st["ctx"].step(u, st["steps"])
    return u


# --------------------------------------------------------------------------- necessary work
def _axis(n, tile, overlap, periodic):
    """(window origin, window length, owner offset, owner length, first owner, whole axis) per tile."""
    out = []
    for t0 in range(0, n, tile):
        t1 = min(n, t0 + tile)
        if periodic and t1 - t0 + 2 * overlap >= n:
            out.append((0, n, t0, t1 - t0, t0, True))
        elif periodic:
            out.append((t0 - overlap, t1 - t0 + 2 * overlap, overlap, t1 - t0, t0, False))
        else:
            lo, hi = max(0, t0 - overlap), min(n, t1 + overlap)
            out.append((lo, hi - lo, t0 - lo, t1 - t0, t0, False))
    return out


def _plan(shape, bc, tile, overlap):
    ax = [_axis(n, t, o, b == "periodic") for n, t, o, b in zip(shape, tile, overlap, bc)]
    return ax if len(ax) == 2 else [[(0, 1, 0, 1, 0, False)], ax[0]]


def _step_work(shape, bc, tile, overlap, prec, steps, shared, cplx=False, builds=0):
    """The apply's multiply-adds; state in and out; the distinct propagators' values, once, or once a
    step where they are more than the 129 MB cache holds; a Pade-13 build's products where the path
    builds (17 of n^3 multiply-adds per phi_1 and operator, with a solve of two right-hand sides)."""
    ys, xs = _plan(shape, bc, tile, overlap)
    npts = shape[0] * (shape[1] if len(shape) > 1 else 1)
    oy, ox = sum(a[3] * a[1] for a in ys), sum(a[3] * a[1] for a in xs)
    mults = oy * ox
    if shared:
        pvals = sum(y[0] * y[2] * x[0] * x[2] for y in {a[1:4] for a in ys} for x in {a[1:4] for a in xs})
    else:
        pvals = mults
    value = {"fp64": 8, "split": 6 if shared else 8, "split_fast": 4}[prec] * (2 if cplx else 1)
    pbytes = pvals * value
    w = (2 if cplx else 1) * 8 * npts
    byts = 2 * w + pbytes * (steps if pbytes > 129e6 else 1) + (0 if shared else 5 * w)
    flops = (8 if cplx else 2) * mults * steps
    if builds:
        cubes = sum((y[1] * x[1]) ** 3 for y in ys for x in xs)
        flops += builds * 17 * 2 * cubes
    return dict(bytes=float(byts), flops=float(flops))


def _case_work(case):
    kind, steps, prec = case["kind"], case["steps"], case["prec"]
    if kind in ("heat1d", "vardiff1d", "schrodinger1d", "porous1d"):
        bc = ("periodic",) if kind == "schrodinger1d" else ("dirichlet",)
        return _step_work((case["n"],), bc, (case["tile"],), (case["overlap"],), prec, steps, kind == "heat1d",
                          cplx=kind == "schrodinger1d", builds=steps if case.get("refresh") else 0)
    if kind == "walls2d":
        return _step_work((case["ny"], case["nx"]), ("dirichlet",) * 2, (case["ty"], case["tx"]),
                          (case["oy"], case["ox"]), prec, steps, True)
    bc = ("periodic",) * 2 if kind == "advdiff2d" else ("dirichlet",) * 2
    return _step_work((case["side"],) * 2, bc, (case["tile"],) * 2, (case["overlap"],) * 2, prec, steps,
                      kind == "advdiff2d", builds=steps if case.get("refresh") else 0)


def work(case):
    if case["kind"] in ("batch", "serve"):
        r, tot = np.random.RandomState(case["pick"] % (1 << 31)), dict(bytes=0.0, flops=0.0)
        for q in range(case["count"]):
            if case["kind"] == "batch":
                side, tile, o, steps, prec = 32 * r.randint(2, case["side_max"] // 32 + 1), int(r.choice([8, 16, 32])), \
                    r.randint(4, 9), case["steps"], case["prec"]
                r.uniform(), r.uniform()
                w = _step_work((int(side),) * 2, ("periodic",) * 2, (tile,) * 2, (int(o),) * 2, prec, steps, True)
            else:
                steps, tol = int(r.randint(1, 21)), 1e-10 if q % 3 == 2 else 1e-6
                if q % 4 == 3:
                    n = int(round(math.exp(r.uniform(math.log(256), math.log(65536)))))
                    w = _step_work((n,), ("dirichlet",), (64,), (16,), "fp64", steps, True)
                else:
                    side = 32 * int(r.randint(4, 17 if tol > 1e-8 else 9))
                    w = _step_work((side,) * 2, ("periodic",) * 2, ((16, 32)[q % 2],) * 2, ((6, 8)[q % 2],) * 2,
                                   "split" if tol > 1e-8 else "fp64", steps, True)
            tot = {k: tot[k] + w[k] for k in tot}
        return tot
    return _case_work(case)


# --------------------------------------------------------------------------- 64-bit results
def _at(c, idx):
    """A coefficient at the window nodes idx: a number stays one."""
    return c.reshape(-1)[idx] if isinstance(c, torch.Tensor) else c


class Windows:
    """All windows of one shape: their mesh nodes, their owners, and X = dt A (+ Jacobian) on them."""

    def __init__(self, p, ys, xs, whole):
        ny, nx = (1,) * (2 - len(p.shape)) + p.shape
        gy = torch.tensor([[(a[0] + i) % ny for i in range(a[1])] for a in ys], device=DEV)
        gx = torch.tensor([[(a[0] + i) % nx for i in range(a[1])] for a in xs], device=DEV)
        idx = gy[:, None, :, None] * nx + gx[None, :, None, :]
        self.idx = idx.reshape(-1, idx.shape[2], idx.shape[3])
        self.own = slice(ys[0][2], ys[0][2] + ys[0][3]), slice(xs[0][2], xs[0][2] + xs[0][3])
        self.whole, self.two = whole, len(p.shape) == 2
        self.c = {k: (_at(v, self.idx) if isinstance(v, torch.Tensor) else v) for k, v in p.coef.items()}
        self.c = {k: v * p.dt for k, v in self.c.items()}
        self.diag = self.cols = None

    def jacobian(self, p, um):
        if p.reaction:
            self.diag = p.dt * (1 - 3 * um.reshape(-1)[self.idx] ** 2)
        if p.porous_m:
            self.cols = p.porous_m * um.reshape(-1)[self.idx].abs() ** (p.porous_m - 1)

    def norm(self):
        big = sum(v.abs().max().item() if isinstance(v, torch.Tensor) else abs(v) for v in self.c.values())
        big += self.diag.abs().max().item() if self.diag is not None else 0.0
        return big * (self.cols.max().item() if self.cols is not None else 1.0)

    def apply(self, v):
        c = self.c
        part = lambda k, s: c[k][s] if isinstance(c[k], torch.Tensor) else c[k]  # noqa: E731
        if self.cols is not None:
            v = v * self.cols
        out = c["C"] * v
        if self.diag is not None:
            out += self.diag * v
        a, l, r = slice(None), slice(1, None), slice(None, -1)
        out[..., l] += part("W", (a, a, l)) * v[..., r]
        out[..., r] += part("E", (a, a, r)) * v[..., l]
        if self.whole[1]:
            out[..., 0] += part("W", (a, a, 0)) * v[..., -1]
            out[..., -1] += part("E", (a, a, -1)) * v[..., 0]
        if self.two:
            out[:, l] += part("S", (a, l)) * v[:, r]
            out[:, r] += part("N", (a, r)) * v[:, l]
            if self.whole[0]:
                out[:, 0] += part("S", (a, 0)) * v[:, -1]
                out[:, -1] += part("N", (a, -1)) * v[:, 0]
        return out

    def act(self, v, phi):
        """phi_1(X) v or exp(X) v by substeps of a Taylor series."""
        sub = max(1, math.ceil(self.norm() / 2.5))
        h = 1.0 / sub
        w = torch.zeros_like(v) if phi else v.clone()
        for _ in range(sub):
            term = (self.apply(w) + v) * h if phi else self.apply(w) * h
            acc = term.clone()
            for k in range(2, 30):
                term = self.apply(term).mul_(h / k)
                acc += term
            w += acc
        return w

    def dense(self, phi):
        """Owner rows of phi_1(X) or exp(X) of the one operator that all these windows share."""
        wy, wx = self.idx.shape[1:]
        n = wy * wx
        X = self.apply(torch.eye(n, device=DEV, dtype=F64).reshape(n, wy, wx)).reshape(n, n).T.contiguous()
        s = max(0, math.ceil(math.log2(max(self.norm(), 1e-3) / 0.5)))
        Y, one = X / 2.0 ** s, torch.eye(n, device=DEV, dtype=F64)
        P = one / math.factorial(15)
        for k in range(14, 0, -1):
            P = Y @ P + one / math.factorial(k)
        E = one + Y @ P
        for _ in range(s):
            P = (E @ P + P) / 2
            E = E @ E
        rows = torch.arange(n, device=DEV).reshape(wy, wx)[self.own].reshape(-1)
        return (P if phi else E)[rows]


def _residual(p, mesh, u):
    """dt F(u) on the whole mesh (one window that is the mesh)."""
    v = u.reshape(mesh.idx.shape)
    if p.porous_m:
        v = v.abs() ** (p.porous_m - 1) * v
    r = mesh.apply(v)
    if p.reaction:
        r = r + p.dt * (v - v ** 3)
    return r.reshape(-1)


def _advance(p, steps):
    phi = p.mode == "phi"
    ys, xs = _plan(p.shape, p.bc, p.tile, p.overlap)
    groups = {}
    for kind in sorted({a[1:4] + a[5:] for a in ys}):
        for kx in sorted({a[1:4] + a[5:] for a in xs}):
            groups[kind, kx] = Windows(p, [a for a in ys if a[1:4] + a[5:] == kind],
                                       [a for a in xs if a[1:4] + a[5:] == kx], (kind[3], kx[3]))
    ny, nx = (1,) * (2 - len(p.shape)) + p.shape
    per = [b == "periodic" for b in p.bc]
    mesh = Windows(p, [(0, ny, 0, ny, 0, False)], [(0, nx, 0, nx, 0, False)], (per[0] and len(per) == 2, per[-1]))
    u = p.u0.reshape(-1).clone()
    shared = len(groups) == 1 and not any(isinstance(v, torch.Tensor) for v in p.coef.values()) and not p.reaction
    shared = shared and not p.porous_m
    P = next(iter(groups.values())).dense(phi) if shared else None
    for k in range(steps):
        if (p.reaction or p.porous_m) and (k == 0 or (p.refresh and k % p.refresh == 0)):
            for w in groups.values():
                w.jacobian(p, u)
        src = _residual(p, mesh, u) if phi else u
        new = u.clone()
        for w in groups.values():
            v = src[w.idx]
            if P is not None:
                y = (v.reshape(v.shape[0], -1) @ P.T).reshape(-1)
            else:
                y = w.act(v, phi)[(slice(None),) + w.own].reshape(-1)
            at = w.idx[(slice(None),) + w.own].reshape(-1)
            new[at] = u[at] + y if phi else y
        u = new
    return u


def exact(case, seed):
    if case["kind"] == "batch":
        return [_advance(p, case["steps"]) for p in _batch(case, seed)]
    if case["kind"] == "serve":
        return [_advance(p, steps).cpu().numpy() for p, _, steps in _requests(case, seed)]
    return _advance(_problem(case, seed), case["steps"])
