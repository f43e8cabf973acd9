"""Propagator builds at the edges of the solve's panels (64 columns), of its groups of panels (256)
and of the products' tiles, against the oracle's Pade-13 (Sec. 3 step 2, Sec. 4): one operator and
several in one batch, windows of one size and clipped ones, FP64 products and tensor-core products.

The bar is that of the other builder tests: a product carries an error below about n 2^-48 (digits) or
n 2^-53 (FP64) of max|A_i,:| max|B_:,j|, and up to a dozen products and the squarings stay within
1e-11 of max|P|."""
import numpy as np
import pytest

from oracle import assemble_operator, decompose, local_propagators
from paper_1505_02248_gb300 import lem as L

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

TOL = 1e-11


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1505_02248_gb300 import build as B
    B.build()
    L.load()


# windows of tile + 2 H nodes
@pytest.mark.parametrize("tile,H", [(31, 1), (32, 16), (33, 16), (95, 16), (97, 16), (223, 16), (224, 16), (225, 16),
                                    (289, 16)])
@pytest.mark.parametrize("prec", ["fp64", "split_fast"])
@pytest.mark.parametrize("mode", ["phi", "exp"])
def test_windows_at_panel_edges(tile, H, prec, mode):
    n = 3 * tile + tile // 2  # (two whole windows, two clipped ones)
    rng = np.random.default_rng(tile)
    k = rng.uniform(0.5, 2.0, n + 1)
    coef = {"C": -(k[:-1] + k[1:]), "W": k[:-1].copy(), "E": k[1:].copy()}
    ctx = L.Lem((n,), ("dirichlet",), coef, 2.0, (tile,), (H,), mode=mode, prec=prec)
    ctx.build()
    X = assemble_operator((n,), ("dirichlet",), coef, 2.0)
    wins = decompose((n,), ("dirichlet",), (tile,), (H,))
    for t in range(len(wins)):
        want = local_propagators(X, wins, mode, tiles=[t])[t]
        got = ctx.propagator(ctx.tile_class(t))
        ni, nl = want.shape
        assert np.abs(got[:ni, :nl] - want).max() <= TOL * np.abs(want).max()
        assert not got[:ni, nl:].any() and not got[ni:].any()
    ctx.close()
