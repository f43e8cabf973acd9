"""The FP64 step without room for its digits (csrc/step_oz.cu): the FP64 GEMM takes over, whether the
propagators' digits are refused at lem_create or the windows' at the first step."""
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


@pytest.mark.parametrize("mode", ["phi", "exp"])
def test_a_step_without_room_for_digits(monkeypatch, mode):
    coef = {"C": -9.5, "W": 3.0, "E": 2.0, "S": 2.5, "N": 2.0}
    shape = (64, 32)  # 32 windows of 256 nodes in one block, 64 owner rows: 16 K blocks of 7 x 2 KB and 7 x 4 KB
    make = lambda: L.Lem(shape, ("periodic",) * 2, coef, 1.0, (8, 8), (4, 4), mode=mode, prec="fp64")  # noqa: E731
    u = np.random.default_rng(1).standard_normal(64 * 32)
    out, held = [], []
    for stage, size in (("create", 16 * 7 * 2048), ("step", 16 * 7 * 4096)):
        if stage == "create":
            monkeypatch.setenv("LEM_FAULT", f"alloc={size}")
        ctx = make()
        monkeypatch.delenv("LEM_FAULT", raising=False)
        ctx.build()
        a, b = torch.tensor(u, device="cuda"), torch.tensor(u, device="cuda")
        monkeypatch.setenv("LEM_FAULT", f"alloc={size}")
        ctx.step(a, 2)
        ctx.sync()
        monkeypatch.delenv("LEM_FAULT")
        ctx.step_noalloc(b, 2)
        torch.cuda.synchronize()
        assert torch.equal(a, b)  # the same kernels
        ctx.step(a, 1)
        ctx.sync()
        out.append(a.cpu().numpy())
        held.append(ctx.info()["device_bytes"])
        ctx.close()
    assert np.array_equal(out[0], out[1]) and held[0] == held[1]


def test_the_servers_estimate_of_a_context():
    """Windows of more than a GiB of digits: what a request's context counts against the budget is what it
    holds, within the scratch of a host state (8 bytes a node)."""
    side = 3872
    coef = {"C": -9.5, "W": 3.0, "E": 2.0, "S": 2.5, "N": 2.0}
    args = ((side, side), ("periodic",) * 2, coef, 1.0, (16, 16), (16, 16))
    ctx = L.Lem(*args, prec="fp64")
    d_u = torch.zeros(side * side, dtype=torch.float64, device="cuda")
    ctx.step(d_u, 1)
    ctx.sync()
    held = ctx.info()["device_bytes"]
    ctx.close()
    srv = L.Server()
    srv.wait(srv.submit(*args, np.zeros(side * side), 1, tol=1e-10), 120.0)
    counted = srv.stats()["device_bytes"]
    srv.close()
    assert held <= counted <= held + 8 * side * side + (32 << 20)
