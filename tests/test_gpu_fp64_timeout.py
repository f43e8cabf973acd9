"""A wait that runs out in the FP64 step on the tensor cores (csrc/step_oz.cu; LEM_FAULT=timeout: the first CTA
arms a stage whose bytes never all come): the host reads LEM_ETIMEOUT, and no owner is written from sums
that are not complete, by one CTA for a unit or by a cluster that shares it."""
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


# windows of 621 nodes (their K blocks shared by a cluster), of 24 nodes (one CTA)
@pytest.mark.parametrize("shape,tile,H", [((95, 92), (19, 23), (2, 2)), ((26, 40), (2, 4), (1, 1))])
def test_an_incomplete_unit_is_not_written(monkeypatch, shape, tile, H):
    rng = np.random.default_rng(0)
    coef = {"C": -4.0, "W": 1.0, "E": 1.0, "S": 1.0, "N": 1.0}
    make = lambda: L.Lem(shape, ("periodic",) * 2, coef, 1.0, tile, H, mode="exp", prec="fp64")  # noqa: E731
    monkeypatch.setenv("LEM_FAULT", "timeout")
    bad = make()
    monkeypatch.delenv("LEM_FAULT")
    good = make()
    info = good.info()
    assert L.APPLY_PATHS[info["apply_path"]] == "fp64_gemm" and info["nclasses"] == 1
    P = rng.uniform(0.5, 1.0, (1, info["n_int"], info["n_loc"]))
    u = rng.uniform(0.5, 1.0, shape[0] * shape[1])
    a, b = torch.tensor(u, device="cuda"), torch.tensor(u, device="cuda")
    for ctx in (bad, good):
        ctx.set_propagators(P)
    good.step(a, 1)
    good.sync()
    bad.step(b, 1)
    with pytest.raises(L.LemError) as e:
        bad.sync()
    assert e.value.status == L.LEM_ETIMEOUT
    bad.sync()  # reported once; the stream is healthy
    new, got = a.cpu().numpy(), b.cpu().numpy()
    kept, written = got == u, got == new
    assert (kept | written).all() and kept.any()
    bad.close()
    good.close()
