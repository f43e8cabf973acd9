"""The batched GEMVs (csrc/step_gemv.cu, csrc/step_band.cu) with loaded propagators of small whole
numbers: every residual, product and partial sum stays below 2^24, so FP32 and FP64 rows alike must
give exactly P R in whole numbers, whatever the order of their sums. Windows whose values fill no whole
16-byte chunk, clipped windows, ragged last tiles, owners that fill no group of rows, and one, two
and three steps (the steps of one call alternate between two buffers on some paths)."""
import numpy as np
import pytest

from oracle import decompose
from paper_1505_02248_gb300 import lem as L

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1505_02248_gb300 import build as B
    B.build()
    L.load()


def _coef(shape, rng, cplx):
    names = "CWE" if len(shape) == 1 else "CWESN"
    n = int(np.prod(shape))
    return {k: rng.integers(-1, 2, n) + (1j * rng.integers(-1, 2, n) if cplx else 0.0) for k in names}


def _residual(u, coef, shape, bc):
    v, r = u.reshape(shape), 0
    get = lambda k: np.reshape(coef[k], shape) if np.ndim(coef[k]) else coef[k]
    for k, axis, d in (("C", 0, 0), ("W", -1, 1), ("E", -1, -1), ("S", 0, 1), ("N", 0, -1)):
        if k not in coef:
            continue
        s = np.roll(v, d, axis)
        if d and bc[axis] == "dirichlet":
            cut = [slice(None)] * len(shape)
            cut[axis] = 0 if d == 1 else shape[axis] - 1
            s[tuple(cut)] = 0
        r = r + get(k) * s
    return np.ravel(r)


def _propagators(ctx, wins, rng, cplx, reach):
    """Per class a few +-1 a row (reach: none further than this many window places from the owner)."""
    info = ctx.info()
    P = np.zeros((info["nclasses"], info["n_int"], info["n_loc"]))
    of = {}
    for t, w in enumerate(wins):
        c = ctx.tile_class(t)
        if c in of:
            continue
        ni, nl = len(w.D), len(w.M)
        A = np.zeros((ni, nl), dtype=complex if cplx else float)
        for i in range(ni):
            lo, hi = (0, nl) if reach is None else (max(0, w.d_pos[i] - reach), min(nl, w.d_pos[i] + reach + 1))
            at = rng.integers(lo, hi, 3)
            if reach is None:
                at[0] = nl - 1 - i % 3  # (the row's last places)
            A[i, at] = rng.choice([-1.0, 1.0], 3)
            if cplx:
                A[i, at] = A[i, at] + 1j * rng.choice([-1.0, 1.0], 3)
        of[c] = A
        if cplx:
            hi, hl = info["n_int"] // 2, info["n_loc"] // 2
            P[c, :ni, :nl], P[c, :ni, hl:hl + nl] = A.real, -A.imag
            P[c, hi:hi + ni, :nl], P[c, hi:hi + ni, hl:hl + nl] = A.imag, A.real
        else:
            P[c, :ni, :nl] = A
    ctx.set_propagators(P)
    return of


def _run(shape, bc, tile, H, prec, steps, path, cplx=False, trunc=False, seed=0):
    rng = np.random.default_rng(seed)
    coef = _coef(shape, rng, cplx)
    ctx = L.Lem(shape, (bc,) * len(shape), coef, 1.0, tile, H, prec=prec)
    if trunc:
        ctx.set_truncation(0.0)
    assert L.APPLY_PATHS[ctx.info()["apply_path"]] == path
    wins = decompose(shape, (bc,) * len(shape), tile, H)
    P = _propagators(ctx, wins, rng, cplx, 3 if trunc else None)
    n = int(np.prod(shape))
    u = rng.integers(-2, 3, n).astype(float)
    if cplx:
        u = u + 1j * rng.integers(-2, 3, n)
    d_u = torch.tensor(u, device="cuda")
    ctx.step(d_u, steps)
    ctx.sync()
    for _ in range(steps):
        r, new = _residual(u, coef, shape, (bc,) * len(shape)), u.copy()
        for t, w in enumerate(wins):
            new[w.D] += P[ctx.tile_class(t)] @ r[w.M]
        u = new
    assert np.abs(u).max() < 2 ** 22
    assert np.array_equal(d_u.cpu().numpy(), u)
    ctx.close()


SHAPES = [((130,), "dirichlet", (20,), (5,)), ((37, 41), "dirichlet", (9, 8), (3, 2)),
          ((48, 70), "periodic", (16, 14), (6, 5)), ((1000,), "dirichlet", (64,), (33,))]


@pytest.mark.parametrize("shape,bc,tile,H", SHAPES)
@pytest.mark.parametrize("prec", ["fp64", "split_fast"])
@pytest.mark.parametrize("steps", [1, 3])
def test_per_tile_propagators(shape, bc, tile, H, prec, steps):
    _run(shape, bc, tile, H, prec, steps, "f32_gemv" if prec == "split_fast" else "fp64_gemv", seed=steps)


@pytest.mark.parametrize("n,tile,H", [(160, 20, 5), (405, 45, 13), (640, 80, 20)])
@pytest.mark.parametrize("prec", ["fp64", "split_fast"])
def test_complex_propagators(n, tile, H, prec):
    _run((n,), "periodic", (tile,), (H,), prec, 2, "f32_gemv" if prec == "split_fast" else "fp64_gemv", cplx=True)


@pytest.mark.parametrize("shape,bc,tile,H", [((130,), "dirichlet", (20,), (5,)), ((3000,), "dirichlet", (64,), (16,)),
                                             ((900,), "periodic", (45,), (11,)), ((31, 45), "dirichlet", (7, 9), (4, 4)),
                                             ((48, 96), "periodic", (24, 32), (4, 4))])
@pytest.mark.parametrize("prec", ["fp64", "split_fast"])
@pytest.mark.parametrize("steps", [1, 2, 3])
def test_truncated_propagators(shape, bc, tile, H, prec, steps):
    _run(shape, bc, tile, H, prec, steps, "f32_band" if prec == "split_fast" else "fp64_band", trunc=True)


# one tile more than half the SMs (one block a tile), a few tiles (many blocks a tile), owners that are no
# multiple of the blocks' rows
@pytest.mark.parametrize("n,tile,H", [(1600, 20, 4), (1024, 64, 16), (300, 100, 20), (340, 85, 9), (51, 17, 4)])
@pytest.mark.parametrize("steps", [2, 3])
def test_steps_of_one_launch(n, tile, H, steps):
    rng = np.random.default_rng(n)
    coef = {"C": -2.0, "W": 1.0, "E": 1.0}
    ctx = L.Lem((n,), ("dirichlet",), coef, 1.0, (tile,), (H,), prec="fp64")
    wins = decompose((n,), ("dirichlet",), (tile,), (H,))
    P = _propagators(ctx, wins, rng, False, None)
    u = rng.integers(-2, 3, n).astype(float)
    d_u = torch.tensor(u, device="cuda")
    ctx.step(d_u, steps)
    ctx.sync()
    for _ in range(steps):
        r, new = _residual(u, coef, (n,), ("dirichlet",)), u.copy()
        for t, w in enumerate(wins):
            new[w.D] += P[ctx.tile_class(t)] @ r[w.M]
        u = new
    assert np.array_equal(d_u.cpu().numpy(), u)
    ctx.close()
