"""The FP64 step on the tensor cores (csrc/step_oz.cu) against exact integer arithmetic.

In EXP mode a step is u_D = P u_M with whatever propagators are loaded, so the digit products can
be checked bit for bit: the digits of P and of each window, the products with s + t <= 6 summed as
integers, one rounding. Sizes cross the tile edges (128 windows, 64 owner rows, 16-node K blocks),
the 128- and 256-node stretches, and the splits of K over a cluster; the values run over a wide
range and include the largest digits."""
import math

import numpy as np
import pytest

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


def _digits(rows):
    """Scale exponents and balanced base-256 digits (7, rows, K) of each row."""
    _, ex = np.frexp(rows)
    e = np.where(rows != 0, ex, -5000).max(axis=1)
    e = np.where(e < -1021, -1022, e)
    N = np.zeros(rows.shape, dtype=object)
    for i in range(rows.shape[0]):
        for k in range(rows.shape[1]):
            x = rows[i, k]
            if x == 0.0:
                continue
            n = int(math.ldexp(abs(math.frexp(x)[0]), 53))  # 53-bit mantissa
            left = math.frexp(x)[1] - 53 + 55 - int(e[i])
            n = n << left if left >= 0 else (n + (1 << (-left - 1))) >> -left
            N[i, k] = -n if x < 0 else n
    d = np.zeros((7,) + rows.shape, dtype=np.int64)
    rest = N.copy()
    for s in range(6, 0, -1):
        q = (rest + 128) % 256 - 128
        d[s] = q.astype(np.int64)
        rest = (rest - q) // 256
    d[0] = rest.astype(np.int64)
    return e, d


def _expected(P, W):
    """P (owners x K) applied to windows W (n x K): the kept levels, rounded once."""
    eP, dP = _digits(P)
    eW, dW = _digits(W)
    T = np.zeros((W.shape[0], P.shape[0]), dtype=object)
    for Lv in range(7):
        S = sum(dW[s] @ dP[Lv - s].T for s in range(Lv + 1))
        T = T + S.astype(object) * (1 << (8 * (6 - Lv)))
    out = np.zeros(T.shape)
    for i in range(T.shape[0]):
        for j in range(T.shape[1]):
            out[i, j] = math.ldexp(float(T[i, j]), int(eW[i]) + int(eP[j]) - 62)
    return out


def _windows(shape, tile, H, u):
    """Windows and owner nodes of a periodic mesh whose tiles divide it."""
    ny, nx = shape
    W, own = [], []
    for y in range(0, ny, tile[0]):
        for x in range(0, nx, tile[1]):
            gy = (np.arange(y - H[0], y + tile[0] + H[0])) % ny
            gx = (np.arange(x - H[1], x + tile[1] + H[1])) % nx
            W.append(u[np.ix_(gy, gx)].ravel())
            own.append((np.arange(y, y + tile[0])[:, None] * nx + np.arange(x, x + tile[1])).ravel())
    return np.array(W), np.array(own)


# (mesh, tile, overlap): 8 windows of 20 nodes; 130 windows (two blocks); 70 owners (two column
# blocks), K 15 x 11 = 165 (a ragged second stretch); K = 256 and 288 exactly; K 621 (a ragged
# third stretch of 256, split over a cluster)
CASES = [((8, 8), (4, 2), (0, 1)), ((26, 40), (2, 4), (1, 1)), ((48, 28), (12, 7), (2, 2)),
         ((64, 32), (8, 8), (4, 4)), ((64, 32), (8, 8), (4, 5)), ((95, 92), (19, 23), (2, 2))]


@pytest.mark.parametrize("shape,tile,H", CASES)
@pytest.mark.parametrize("values", ["wide", "extreme"])
def test_step_is_the_rounded_integer_sum(shape, tile, H, values):
    rng = np.random.default_rng(sum(shape) + len(values))
    coef = {"C": -4.0, "W": 1.0, "E": 1.0, "S": 1.0, "N": 1.0}
    ctx = L.Lem(shape, ("periodic", "periodic"), coef, 0.1, tile, H, mode="exp", prec="fp64")
    info = ctx.info()
    assert L.APPLY_PATHS[info["apply_path"]] == "fp64_gemm" and info["nclasses"] == 1
    n_int, n_loc = info["n_int"], info["n_loc"]
    if values == "wide":
        P = rng.standard_normal((1, n_int, n_loc)) * np.exp2(rng.integers(-40, 3, (1, n_int, n_loc)))
        u = rng.standard_normal(shape) * np.exp2(rng.integers(-70, 1, shape))
        u[rng.random(shape) < 0.1] = 0.0
    else:  # digits 128, -128, -128, ...: every product at the bound, levels of one sign
        big = float(2 ** 55 - 128 * sum(256 ** k for k in range(6))) * 2.0 ** -55
        P = np.full((1, n_int, n_loc), big)
        u = np.full(shape, -big)
    ctx.set_propagators(P)
    W, own = _windows(shape, tile, H, u)
    want = np.zeros(u.size)
    want[own] = _expected(P[0], W)
    d_u = torch.tensor(u.ravel(), device="cuda")
    ctx.step(d_u, 1)
    ctx.sync()
    assert np.array_equal(d_u.cpu().numpy(), want)


def test_non_finite_values_reach_the_same_owners_as_in_fp64():
    shape, tile, H = (64, 64), (8, 8), (3, 3)
    coef = {"C": -4.0, "W": 1.0, "E": 1.0, "S": 1.0, "N": 1.0}
    u = np.random.default_rng(3).standard_normal(shape)
    u[5, 9], u[40, 41] = np.inf, np.nan
    for mode in ("phi", "exp"):
        ctx = L.Lem(shape, ("periodic", "periodic"), coef, 0.5, tile, H, mode=mode, prec="fp64")
        ctx.build()
        got = torch.tensor(u.ravel(), device="cuda")
        ctx.step(got, 1)
        ctx.sync()
        plain = torch.tensor(u.ravel(), device="cuda")
        ctx.step_noalloc(plain, 1)  # the FP64 multiply-add path
        torch.cuda.synchronize()
        a, b = got.cpu().numpy(), plain.cpu().numpy()
        assert np.array_equal(np.isnan(a), np.isnan(b)) and np.array_equal(np.isposinf(a), np.isposinf(b))
        ok = np.isfinite(b)
        assert ok.sum() > 0.8 * ok.size
        # both sides carry at most about K 2^-53 of sum |P| |u| ~ 196 x 2^-53 x 10
        assert np.abs(a[ok] - b[ok]).max() <= 1e-12


def test_walls_ragged_tiles_and_split_agree_with_the_plain_path():
    """Classes of unlike window sizes in one launch, against the FP64 multiply-add path."""
    rng = np.random.default_rng(5)
    coef = {"C": -9.5, "W": 3.0, "E": 2.0, "S": 2.5, "N": 2.0}
    for mode in ("phi", "exp"):
        for shape, tile, H in (((131, 117), (9, 12), (4, 5)), ((700,), (20,), (9,))):
            co = coef if len(shape) == 2 else {k: coef[k] for k in "CWE"}
            ctx = L.Lem(shape, ("dirichlet",) * len(shape), co, 1.0, tile, H, mode=mode, prec="fp64")
            ctx.build()
            assert L.APPLY_PATHS[ctx.info()["apply_path"]] == "fp64_gemm"
            u = rng.standard_normal(shape).ravel()
            a, b = torch.tensor(u, device="cuda"), torch.tensor(u, device="cuda")
            ctx.step(a, 3)
            ctx.sync()
            ctx.step_noalloc(b, 3)
            torch.cuda.synchronize()
            assert torch.linalg.norm(a - b) <= 1e-13 * torch.linalg.norm(b)
