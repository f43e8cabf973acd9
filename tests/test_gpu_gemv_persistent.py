"""Steps of small problems in one launch (csrc/step_gemv.cu, gemv_persistent_kernel), with loaded propagators of small
whole numbers: exact whatever the order of the sums. A tile's rows shared over many blocks, a block a
tile, propagators in shared memory or read from global memory, and more tiles than the device holds
blocks at once, FP32 rows with four and with five blocks an SM."""
import numpy as np
import pytest

from oracle import decompose
from paper_1505_02248_gb300 import lem as L
from test_gpu_gemv import _propagators, _residual

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1505_02248_gb300 import build as B
    B.build()
    L.load()


# 3 and 16 tiles (shared), 80 (a block each, in shared memory), windows of 1100 nodes, 640 tiles (two rounds), 2000 and
# 1900 (FP32 rows with five blocks an SM: three rounds instead of four)
@pytest.mark.parametrize("n,tile,H", [(300, 100, 20), (1024, 64, 16), (1600, 20, 4), (3300, 300, 400), (6400, 10, 3),
                                      (8000, 4, 2), (7600, 4, 1)])
@pytest.mark.parametrize("prec", ["fp64", "split_fast"])
@pytest.mark.parametrize("steps", [2, 3])
def test_steps_of_one_launch(n, tile, H, prec, steps):
    rng = np.random.default_rng(n)
    coef = {"C": np.full(n, -2.0), "W": np.full(n, 1.0), "E": np.full(n, 1.0)}  # (node by node: a class a tile)
    ctx = L.Lem((n,), ("dirichlet",), coef, 1.0, (tile,), (H,), prec=prec)
    assert L.APPLY_PATHS[ctx.info()["apply_path"]] == ("f32_gemv" if prec == "split_fast" else "fp64_gemv")
    wins = decompose((n,), ("dirichlet",), (tile,), (H,))
    P = _propagators(ctx, wins, rng, False, None)
    u = rng.integers(-2, 3, n).astype(float)
    d_u = torch.tensor(u, device="cuda")
    ctx.set_timing(True)
    ctx.step(d_u, steps)
    ctx.sync()
    assert ctx.get_timing()[1] == 1  # launches
    for _ in range(steps):
        r, new = _residual(u, coef, (n,), ("dirichlet",)), u.copy()
        for t, w in enumerate(wins):
            new[w.D] += P[ctx.tile_class(t)][:len(w.D), :len(w.M)] @ r[w.M]
        u = new
    assert np.array_equal(d_u.cpu().numpy(), u)
    ctx.close()
