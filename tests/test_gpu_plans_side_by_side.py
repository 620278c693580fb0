"""Plans of different footprints alive at once: an older plan with the larger
footprint keeps working after a smaller one is created and used, in every
form (the shared-memory attribute belongs to a kernel, not to a plan).  The
same call before and after gives the same image up to the order of the FP64
sums."""
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


@pytest.mark.parametrize("n,rows,kw", [
    (128, 65, dict(path="fused")), (128, 99, dict(path="fused")), (128, 41, dict(path="piped")),
    (256, 121, dict(path="cluster")), (256, 121, dict(precision="fp16")), (256, 121, dict(precision="bf16")),
    (256, 121, dict(path="unfused")), (256, 121, dict(path="unfused", batch_persistent=True)),
    (128, 65, dict(path="unfused")),
])
def test_older_plan(n, rows, kw):
    from paper_1603_02126_gb300 import Plan
    rng = np.random.default_rng(rows)
    cell_m = 0.5 * 299792458.0 / 50e6
    out = []

    def plan(rows, na):
        h = ((rows - 3) / 2 - 0.02) * cell_m
        ant = rng.uniform(-h, h, (na, 2))
        ant[0], ant[1] = (-h, -h), (h, h)
        p = Plan(ant, [50e6, 49e6], n, 0.5, **kw)
        return p, torch.from_numpy(rng.integers(0, 256, (9, 2, na), dtype=np.uint8)).cuda()

    a, va = plan(rows, 200)
    out.append(a.image(va))
    b, vb = plan(9, 20)
    b.image(vb)
    out.append(a.image(va))
    assert a.sync() == 0 and b.sync() == 0
    assert torch.linalg.norm(out[1] - out[0]) <= 1e-12 * torch.linalg.norm(out[0])
