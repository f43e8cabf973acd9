"""Accuracy of the FP64 step on the tensor cores (csrc/step_oz.cu), element by element.

In EXP mode a step is u_D = P u_M, so each owner can be compared with its exact sum. FP64
multiply-adds give it within K 2^-53 sum_k |P_k| |u_k|. A digit sum's error goes with the largest
values instead: at most K (2^-53.4 + 2^-55) 2^(e + f), 2^(e + f) <= 4 max|P| max|u|. Digits are used
where sum_k |P_k| |u_k| >= 2^-2 2^(e + f), so that every owner is within 4.1 K 2^-53 sum_k |P_k| |u_k|,
whatever the range of the window's or the row's values."""
import numpy as np
import pytest

from paper_1505_02248_gb300 import lem as L

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

LD = np.longdouble
HEAT1 = {"C": -20.0, "W": 10.0, "E": 10.0}
HEAT2 = {"C": -9.5, "W": 3.0, "E": 2.0, "S": 2.5, "N": 2.0}


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1505_02248_gb300 import build as B
    B.build()
    L.load()


def _periodic(shape, tile, H, coef, mode="exp"):
    ctx = L.Lem(shape, ("periodic",) * len(shape), coef, 1.0, tile, H, mode=mode, prec="fp64")
    assert L.APPLY_PATHS[ctx.info()["apply_path"]] == "fp64_gemm" and ctx.info()["nclasses"] == 1
    return ctx


def _windows(shape, tile, H, pick=None):
    """Node numbers of windows and owners of a periodic mesh whose tiles divide it."""
    sh, ti, ov = ((1,) + tuple(v) if len(shape) == 1 else tuple(v) for v in (shape, tile, H))
    if len(shape) == 1:
        ov = (0, ov[1])
    M, D = [], []
    starts = [(y, x) for y in range(0, sh[0], ti[0]) for x in range(0, sh[1], ti[1])]
    for y, x in (starts if pick is None else [starts[q] for q in pick]):
        gy, gx = np.arange(y - ov[0], y + ti[0] + ov[0]) % sh[0], np.arange(x - ov[1], x + ti[1] + ov[1]) % sh[1]
        M.append((gy[:, None] * sh[1] + gx).ravel())
        D.append((np.arange(y, y + ti[0])[:, None] * sh[1] + np.arange(x, x + ti[1])).ravel())
    return np.array(M), np.array(D)


def _check(got, P, u, M, D):
    W = u[M]
    want = W.astype(LD) @ P.T.astype(LD)
    size = (np.abs(W).astype(LD) @ np.abs(P).T.astype(LD))
    err = np.abs(got[D].astype(LD) - want)
    # (and 2^-1074 a term where values are subnormal)
    assert (err <= 4.1 * P.shape[1] * LD(2) ** -53 * size + P.shape[1] * LD(2) ** -1074).all()


def _field(kind, shape, rng):
    x = np.stack(np.meshgrid(*[np.arange(n) for n in shape], indexing="ij"))
    mid = np.array(shape).reshape((-1,) + (1,) * len(shape)) * 0.4
    d2 = ((x - mid) ** 2).sum(0)
    if kind == "bump":  # a narrow bump, its values in a window many orders of magnitude apart
        return np.exp(-d2 / 40.0)
    if kind == "patch":  # zero away from a patch, whole windows of zeros, some subnormal values
        return np.where(d2 < 60, 1.0 + rng.random(shape), np.where(rng.random(shape) < 0.02, 3e-310, 0.0))
    if kind == "tiny":  # small enough that digits would cut subnormal values
        return rng.standard_normal(shape) * 1e-305
    if kind == "smooth":
        return np.sin(2 * np.pi * x[-1] / shape[-1]) * np.cos(2 * np.pi * x[0] / shape[0])
    return rng.standard_normal(shape) * np.exp2(rng.integers(-70, 1, shape))


# K 96 (many windows), 16 x 16 = 256, and 23 x 27 = 621 (split over a cluster)
GEOM = [((64 * 40,), (64,), (16,), HEAT1), ((64, 32), (8, 8), (4, 4), HEAT2), ((95, 92), (19, 23), (2, 2), HEAT2)]


@pytest.mark.parametrize("shape,tile,H,coef", GEOM)
@pytest.mark.parametrize("kind", ["bump", "patch", "tiny", "smooth", "wide"])
@pytest.mark.parametrize("rows", ["built", "loaded"])
def test_owners_keep_the_accuracy_of_multiply_adds(shape, tile, H, coef, kind, rows):
    rng = np.random.default_rng(len(kind) + shape[0])
    ctx = _periodic(shape, tile, H, coef)
    info = ctx.info()
    if rows == "built":
        ctx.build()
        P = ctx.propagator(0)
    else:  # rows over a wide range, with few values, with none, of small values
        P = rng.standard_normal((info["n_int"], info["n_loc"])) * np.exp2(rng.integers(-40, 3, (info["n_int"], info["n_loc"])))
        P[1] = 0.0
        P[2] = np.where(rng.random(info["n_loc"]) < 0.15, P[2], 0.0)
        P[3] *= 1e-300
        ctx.set_propagators(P[None])
    u = _field(kind, shape, rng).ravel()
    M, D = _windows(shape, tile, H)
    d_u = torch.tensor(u, device="cuda")
    ctx.step(d_u, 1)
    ctx.sync()
    _check(d_u.cpu().numpy(), P, u, M, D)
    ctx.close()


@pytest.mark.parametrize("shape,tile,H,coef", GEOM)
def test_a_bumps_residual_is_propagated_as_by_multiply_adds(shape, tile, H, coef):
    """PHI mode, against the FP64 multiply-add path: both carry at most the bound above, and a
    rounding of the updated owner."""
    rng = np.random.default_rng(1)
    ctx = _periodic(shape, tile, H, coef, mode="phi")
    ctx.build()
    P, u = ctx.propagator(0), _field("bump", shape, rng).ravel()
    a, b = torch.tensor(u, device="cuda"), torch.tensor(u, device="cuda")
    ctx.step(a, 1)
    ctx.sync()
    ctx.step_noalloc(b, 1)
    torch.cuda.synchronize()
    v = u.reshape(shape)
    r = coef["C"] * v
    for k, (axis, by) in {"W": (-1, 1), "E": (-1, -1), "S": (0, 1), "N": (0, -1)}.items():
        r = r + coef[k] * np.roll(v, by, axis) if k in coef else r
    M, D = _windows(shape, tile, H)
    size = np.abs(r.ravel()[M]) @ np.abs(P).T
    got, ref = a.cpu().numpy()[D], b.cpu().numpy()[D]
    assert (np.abs(got - ref) <= 5.1 * P.shape[1] * 2.0 ** -53 * 1.01 * size + 2.0 ** -52 * np.abs(ref)).all()
    ctx.close()


def _dense(rng, shape):
    """Values of one binade and either sign: sum |P| |u| is never small."""
    return rng.uniform(0.5, 1.0, shape) * rng.choice([-1.0, 1.0], shape)


def _digits(rows):
    _, ex = np.frexp(rows)
    e = ex.max(axis=1)
    v = np.ldexp(rows, 55 - e[:, None])
    N = (np.sign(v) * np.floor(np.abs(v) + 0.5)).astype(np.int64)
    d = np.zeros((7,) + rows.shape)
    for s in range(6, 0, -1):
        q = (N + 128) % 256 - 128
        d[s], N = q, (N - q) // 256
    d[0] = N
    return e, d


def _digit_sums(P, W):
    """The kept levels' whole-number sums, rounded once."""
    (eP, dP), (eW, dW) = _digits(P), _digits(W)
    S = [sum(dW[s] @ dP[lv - s].T for s in range(lv + 1)) for lv in range(7)]  # (below 2^53: exact)
    hi = sum(S[lv].astype(np.int64) << (8 * (3 - lv)) for lv in range(4))
    lo = sum(S[lv].astype(np.int64) << (8 * (6 - lv)) for lv in range(4, 7))
    H, R = hi + (lo >> 24), lo & 0xFFFFFF
    assert (np.abs(H) < 1 << 51).all()
    return np.ldexp(H.astype(float) + np.ldexp(R.astype(float), -24), eW[:, None] + eP[None, :] - 38)


# 4096 windows in 32 blocks; 54 blocks of 3 column blocks each, more units than SMs; two groups of windows
# (more than 1 GiB of digits), of 5184 nodes
@pytest.mark.parametrize("shape,tile,H,pick", [((256, 256), (4, 4), (1, 1), 400), ((984, 984), (12, 12), (1, 1), 300),
                                               ((2032, 2032), (16, 16), (28, 28), 24)])
def test_dense_rows_are_the_rounded_digit_sums(shape, tile, H, pick):
    rng = np.random.default_rng(shape[0])
    ctx = _periodic(shape, tile, H, HEAT2)
    info = ctx.info()
    P = _dense(rng, (info["n_int"], info["n_loc"]))
    ctx.set_propagators(P[None])
    u = _dense(rng, shape).ravel()
    n = info["ntiles"]
    q = np.unique(np.concatenate([[0, 1, n // 2, n - 2, n - 1], rng.integers(0, n, pick)]))
    M, D = _windows(shape, tile, H, q)
    d_u = torch.tensor(u, device="cuda")
    ctx.step(d_u, 1)
    ctx.sync()
    assert np.array_equal(d_u.cpu().numpy()[D], _digit_sums(P, u[M]))
    ctx.close()


def test_unlike_classes_are_the_rounded_digit_sums():
    """Walls and ragged tiles: windows of 25 to 1156 nodes, more units than SMs, so a CTA goes from one
    number of K blocks to another."""
    from oracle import decompose
    shape, tile, H = (983, 611), (24, 22), (5, 5)
    ctx = L.Lem(shape, ("dirichlet",) * 2, HEAT2, 1.0, tile, H, mode="exp", prec="fp64")
    info = ctx.info()
    assert L.APPLY_PATHS[info["apply_path"]] == "fp64_gemm" and info["nclasses"] > 8
    rng = np.random.default_rng(0)
    P = _dense(rng, (info["nclasses"], info["n_int"], info["n_loc"]))
    ctx.set_propagators(P)
    u = _dense(rng, shape).ravel()
    d_u = torch.tensor(u, device="cuda")
    ctx.step(d_u, 1)
    ctx.sync()
    got = d_u.cpu().numpy()
    seen = {}
    for t, w in enumerate(decompose(shape, ("dirichlet",) * 2, tile, H)):
        c = ctx.tile_class(t)
        if seen.setdefault(c, 0) < 6:
            seen[c] += 1
            assert np.array_equal(got[w.D], _digit_sums(P[c][:len(w.D), :len(w.M)], u[w.M][None])[0])
    ctx.close()
