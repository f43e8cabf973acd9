"""Contexts beside others in one process: the shared memory that one's kernels take does not bound the other's, and
a context on a stream of its own does not wait for work on the legacy stream."""
import time

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


@pytest.mark.parametrize("tol", [None, 0.0])
def test_a_second_context_with_smaller_windows(tol):
    """Windows above 48 KB of shared memory (7200 and 6600 nodes), dense rows and boxes."""
    def make(shape):
        n, tile = shape[0] * shape[1], (shape[0] // 4, shape[1])
        coef = {"C": -4.0, "W": 1.0, "E": 1.0, "S": 1.0, "N": 1.0}
        ctx = L.Lem(shape, ("dirichlet",) * 2, coef, 1.0, tile, shape, mode="exp", prec="fp64")
        info = ctx.info()
        assert info["n_loc"] == n and info["nclasses"] == 4
        P = np.zeros((4, n // 4, n))  # each owner takes the value of the node before it
        for c in range(4):
            i = np.arange(n // 4)
            at = c * (n // 4) + i - 1
            P[c, i[at >= 0], at[at >= 0]] = 1.0
        ctx.set_propagators(P)
        if tol is not None:
            ctx.set_truncation(tol)
        assert L.APPLY_PATHS[ctx.info()["apply_path"]] == ("fp64_gemv" if tol is None else "fp64_band")
        return ctx

    def check(ctx, shape):
        u = np.random.default_rng(shape[0]).standard_normal(shape[0] * shape[1])
        d_u = torch.tensor(u, device="cuda")
        ctx.step(d_u, 1)
        ctx.sync()
        assert np.array_equal(d_u.cpu().numpy(), np.concatenate([[0.0], u[:-1]]))

    large = make((80, 90))
    check(large, (80, 90))
    small = make((60, 110))
    check(small, (60, 110))
    check(large, (80, 90))
    large.close()
    small.close()


@pytest.mark.parametrize("prec", ["fp64", "split"])
def test_sync_waits_for_the_contexts_stream_only(prec):
    st = torch.cuda.Stream()
    coef = {"C": -46.0, "W": 14.0, "E": 10.0, "S": 12.0, "N": 10.0}
    ctx = L.Lem((64, 64), ("periodic",) * 2, coef, 0.1, (8, 8), (4, 4), prec=prec, stream=st.cuda_stream)
    assert L.APPLY_PATHS[ctx.info()["apply_path"]] == ("fp64_gemm" if prec == "fp64" else "tc_split")
    ctx.build()
    u = torch.ones(64 * 64, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    ctx.step(u, 1)
    ctx.sync()
    torch.cuda._sleep(2_000_000_000)  # about a second on the legacy stream
    t0 = time.perf_counter()
    ctx.step(u, 1)
    ctx.sync()
    took = time.perf_counter() - t0
    torch.cuda.synchronize()
    whole = time.perf_counter() - t0
    assert whole > 0.5 and took < 0.5 * whole
    ctx.close()
