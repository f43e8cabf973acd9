"""The solve of the propagator build, panel by panel (csrc/builder.cu, solve_gj)."""
import threading

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


@pytest.mark.parametrize("tile,H", [(8, 4), (16, 4), (16, 6)])
def test_one_operator_is_built_alike_for_every_apply(tile, H):
    """One operator for all windows (the tensor-core split apply) and the same coefficients node by node (a
    propagator per tile, FP32 rows): the windows' matrices are the same, and so are the builds, bit for
    bit: neither takes products that round worse."""
    side = 4 * tile
    coef = {"C": -46.0, "W": 14.0, "E": 10.0, "S": 12.0, "N": 10.0}
    one = L.Lem((side, side), ("periodic",) * 2, coef, 1.0, (tile,) * 2, (H,) * 2, prec="split")
    per = L.Lem((side, side), ("periodic",) * 2, {k: np.full(side * side, v) for k, v in coef.items()}, 1.0, (tile,) * 2,
                (H,) * 2, prec="split_fast")
    assert L.APPLY_PATHS[one.info()["apply_path"]] == "tc_split" and L.APPLY_PATHS[per.info()["apply_path"]] == "f32_gemv"
    one.build()
    per.build()
    P = one.propagator(0)
    for c in (0, 5, 15):
        assert np.array_equal(per.propagator(c), P)
    one.close()
    per.close()


@pytest.mark.parametrize("prec", ["fp64", "split_fast"])
def test_a_build_out_of_scratch_half_way(monkeypatch, prec):
    """The elimination's scratch is refused when the products before it are already on their way: the build
    reports it, and others, on another stream too, are not disturbed."""
    coef = {"C": -2.0, "W": 1.0, "E": 1.0}
    n = 700 + 2 * 40
    make = lambda: L.Lem((2800,), ("periodic",), coef, 1.0, (700,), (40,), prec=prec,  # noqa: E731
                         stream=torch.cuda.Stream().cuda_stream)
    good = make()
    good.build()
    want = good.propagator(0)
    for k in range(6):
        bad, other = make(), make()
        monkeypatch.setenv("LEM_FAULT", f"alloc={n * 64 * 8}")  # the panel's tracker
        with pytest.raises(L.LemError) as e:
            bad.build()
        assert e.value.status == L.LEM_ENOMEM
        monkeypatch.delenv("LEM_FAULT")
        other.build()
        assert np.array_equal(other.propagator(0), want)
        bad.build()
        assert np.array_equal(bad.propagator(0), want)
        bad.close()
        other.close()
    good.close()


def test_builds_of_unlike_windows_in_threads():
    """The panel kernel's shared memory follows the window: builds of large and small windows at once,
    each on a stream of its own, do not disturb each other."""
    coef = {"C": -2.0, "W": 1.0, "E": 1.0}
    sizes = [(1000, 40), (200, 20), (216, 20), (280, 20)]  # windows of 1080, 240, 256 and 320 nodes
    failed, want = [], []
    ctxs = [L.Lem((4 * t,), ("periodic",), coef, 1.0, (t,), (h,), prec="split", stream=torch.cuda.Stream().cuda_stream)
            for t, h in sizes]
    for c in ctxs:
        c.build()
        want.append(c.propagator(0))
    done = threading.Event()

    def work(k, more):
        try:
            while more():
                ctxs[k].build()
            if not np.array_equal(ctxs[k].propagator(0), want[k]):
                failed.append("other propagators")
        except L.LemError as e:
            failed.append(str(e))

    left = iter([True] * 100 + [False])
    small = [threading.Thread(target=work, args=(k, lambda: not done.is_set())) for k in (1, 2, 3)]
    for t in small:
        t.start()
    work(0, lambda: next(left))
    done.set()
    for t in small:
        t.join()
    assert not failed
    for c in ctxs:
        c.close()


def test_scratch_kept_by_refreshing_contexts_is_bounded():
    """Each keeps the scratch of its builds (about 3 GB here) while all of them together stay within 16 GiB;
    what one gives back another may keep."""
    side = 80
    rng = np.random.default_rng(0)
    h = 1.0 / (side + 1)
    k = rng.uniform(0.5, 2.0) / h ** 2
    coef = {"C": np.full(side * side, -4 * k), **{w: np.full(side * side, k) for w in "WESN"}}
    u = torch.tensor(rng.standard_normal(side * side), device="cuda")
    ctxs = [L.Lem((side, side), ("dirichlet",) * 2, coef, 2.0 / k, (16, 16), (6, 6), prec="split", reaction=True, refresh=1)
            for _ in range(7)]
    bare = [c.info()["device_bytes"] for c in ctxs]

    def kept(c):
        ctxs[c].build(u)
        return ctxs[c].info()["device_bytes"] - bare[c]

    held = [kept(c) for c in range(7)]
    want = ctxs[0].propagator(3)
    assert 1 << 30 < held[0] <= 4 << 30 and held[-1] == 0
    assert sum(held) <= 16 << 30
    ctxs[0].close()
    assert kept(6) == held[1]
    assert np.array_equal(ctxs[6].propagator(3), want) and np.array_equal(ctxs[5].propagator(3), want)
    for c in ctxs[1:]:
        c.close()


@pytest.mark.parametrize("prec", ["fp64", "split_fast"])
def test_windows_beyond_the_panel_kernel(prec):
    """Windows of more than 2880 nodes, whose panels do not fit a cluster's shared memory, are eliminated
    column by column: one window that is the line, against the sine modes of its Laplacian. The bar is that
    of the other builder tests, 1e-11 of max|P|."""
    n, mu = 2901, 2.0  # (the last panel is ragged)
    ctx = L.Lem((n,), ("dirichlet",), {"C": -2 * mu, "W": mu, "E": mu}, 1.0, (n,), (0,), prec=prec)
    assert ctx.info()["n_loc"] == n
    ctx.build()
    P = ctx.propagator(0)
    ctx.close()
    j = np.arange(1, n + 1)
    lam = -4 * mu * np.sin(np.pi * j / (2 * (n + 1))) ** 2
    S = np.sin(np.pi * np.outer(j, j) / (n + 1))
    want = (S * (np.expm1(lam) / lam)) @ S * (2 / (n + 1))
    assert np.abs(P - want).max() <= 1e-11 * np.abs(want).max()
