"""epic_autotune of plans that image frame pairs through device memory tunes
the batch length, which is all they read, and leaves the other parameters,
which shape other calls of the plan, as they were."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__
    __graft_entry__.build()


@pytest.mark.parametrize("n,path,units,cols", [(128, "fused", 4, 4), (256, "unfused", 4, 4)])
def test_parameters(n, path, units, cols):
    from paper_1603_02126_gb300 import Plan
    rng = np.random.default_rng(n)
    ant = rng.uniform(-143.0, 143.0, (60, 2))
    p = Plan(ant, [50e6, 49e6], n, 0.5, path=path)
    v = torch.from_numpy(rng.integers(0, 256, (300, 2, 60), dtype=np.uint8)).cuda()
    ref = p.image(v).clone()
    r = p.autotune(v)
    assert r["units_target"] == units and r["cols_target"] == cols
    assert r["candidates"] >= 1
    assert r["batch_time"] == 0 or (r["batch_time"] % 2 == 0 and 2 <= r["batch_time"] < 300)
    assert 0 < r["ms_best"] <= r["ms_default"]
    img = p.image(v)
    assert torch.linalg.norm(img - ref) <= 1e-6 * torch.linalg.norm(ref)       # FP32 runs of another length
