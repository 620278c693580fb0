"""Scratch of fused plans that image through the wide form (N = 128, large
footprints): held from creation, so that image calls allocate nothing, run
inside a stream capture without a call before it, and leave a captured graph
valid whatever is imaged in between."""
import numpy as np
import pytest

import epic_synth as synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__
    __graft_entry__.build()


def _plan(stream, C=3, na=90, workspace_bytes=0):
    from paper_1603_02126_gb300 import Plan
    rng = np.random.default_rng(7)
    cell_m = 0.5 * 299792458.0 / 50e6
    h = 48.4 * cell_m
    ant = rng.uniform(-h, h, (na, 2))
    ant[0], ant[1] = (-h, -h), (h, h)
    freqs = np.linspace(50e6, 48e6, C)
    p = Plan(ant, freqs, 128, 0.5, path="fused", stream=stream.cuda_stream, workspace_bytes=workspace_bytes)
    sky = np.array([[0.0, 0.0, 5.0], [0.17, -0.11, 1.0]])
    p.configure((0.0, 0.0), sky, 0.5, g0=synth.true_gains(C, na, rng))
    return p


def _volt(T, C=3, na=90, seed=1):
    g = torch.Generator().manual_seed(seed)
    return torch.randint(0, 256, (T, C, na), dtype=torch.uint8, generator=g).cuda()


def _close(a, b):
    return torch.linalg.norm(a - b) / torch.linalg.norm(b) <= 1e-12      # FP64 sums in another order


def test_graph_survives_longer_calls():
    st = torch.cuda.Stream()
    p = _plan(st)
    v, big = _volt(128), _volt(2000, seed=2)
    img, other = (torch.zeros((3, 128, 128), dtype=torch.float64, device="cuda") for _ in range(2))
    torch.cuda.synchronize()
    p.image(v, img)
    p.sync()
    ref, g0 = img.clone(), p.gains()
    p.update()
    p.set_gains(g0)
    p.graph_capture(v, img)
    p.image(big, other)
    p.update()
    p.set_gains(g0)
    p.graph_launch()
    assert p.sync() == 0
    assert _close(img, ref)


@pytest.mark.parametrize("budget", [0, 3 * 2 * 128 * 100 * 8])
def test_image_calls_allocate_nothing(budget):
    st = torch.cuda.Stream()
    p = _plan(st, workspace_bytes=budget)
    img = torch.zeros((3, 128, 128), dtype=torch.float64, device="cuda")
    volts = [_volt(T) for T in (2, 128, 2000)]
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    for v in volts:
        p.image(v, img)
    torch.cuda.synchronize()
    assert p.info()["batch_time"] > 0                         # the wide form ran
    assert torch.cuda.mem_get_info()[0] == free


def test_first_call_inside_a_capture():
    st = torch.cuda.Stream()
    p, q = _plan(st), _plan(st)
    v = _volt(77)
    img, ref = (torch.zeros((3, 128, 128), dtype=torch.float64, device="cuda") for _ in range(2))
    torch.cuda.synchronize()
    q.image(v, ref)
    q.sync()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=st):
        p.image(v, img)
    graph.replay()
    torch.cuda.synchronize()
    assert p.info()["batch_time"] > 0
    assert _close(img, ref)
