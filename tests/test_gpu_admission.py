"""Admission of the FP64 tier (csrc/server.cpp): it leaves a quarter of the budget to the split tier, but a
request that needs more than the other three runs where nothing else does."""
import numpy as np
import pytest

from paper_1505_02248_gb300 import lem as L
from paper_1505_02248_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1505_02248_gb300 import build as B
    B.build()
    L.load()


def test_a_request_of_more_than_three_quarters_of_the_budget():
    srv = L.Server(budget_bytes=int(66e6))  # (a context with its build's scratch: about 58 MB)
    done = []
    for k in range(2):
        wl = W.advdiff2d(side=256, tile=16, overlap=4, ell=8.0, dt=1.0 + 0.5 * k, seed=20 + k)
        st = wl["u0"].copy()
        done.append((wl, st, srv.submit(wl["shape"], wl["bc"], wl["coef"], wl["dt"], wl["tile"], wl["overlap"], st, 3, 1e-10)))
    for wl, st, t in done:
        srv.wait(t, 20.0)
        ctx = L.Lem.from_workload(wl, prec="fp64")
        u = torch.tensor(wl["u0"], device="cuda")
        ctx.step(u, 3)
        ctx.sync()
        assert np.array_equal(st, u.cpu().numpy())
        ctx.close()
    srv.close()
