"""Buffers that a captured call holds stay valid when later calls outgrow
them: a plan's own graph on the unfused path and in the multiple-pixel form,
and a caller's capture of the X-engine.  A replay after longer calls gives
what it gave before them."""
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


C, NA = 2, 48


def _plan(n, stream, **kw):
    from paper_1603_02126_gb300 import Plan
    rng = np.random.default_rng(11)
    ant = rng.uniform(-15.0, 15.0, (NA, 2))
    p = Plan(ant, np.array([50e6, 48e6]), n, 0.5, stream=stream.cuda_stream, **kw)
    p.configure((0.0, 0.0), np.array([[0.0, 0.0, 5.0], [0.17, -0.11, 1.0]]), 0.5, g0=synth.true_gains(C, NA, rng))
    return p


def _volt(T, seed):
    g = torch.Generator().manual_seed(seed)
    return torch.randint(0, 256, (T, C, NA), dtype=torch.uint8, generator=g).cuda()


def _same(a, b):
    return torch.linalg.norm(a - b) / torch.linalg.norm(b) <= 1e-12      # FP64 sums in another order


@pytest.mark.parametrize("n,path,pixels", [(256, "unfused", False), (128, "unfused", False), (64, "fused", True)])
def test_plan_graph(n, path, pixels):
    st = torch.cuda.Stream()
    p = _plan(n, st, path=path)
    if pixels:
        p.configure_pixels([[0.0, 0.0], [0.17, -0.11]])
    v = _volt(40, 1)
    img, other = (torch.zeros((C, n, n), dtype=torch.float64, device="cuda") for _ in range(2))
    gout = torch.zeros((C, NA), dtype=torch.complex128, device="cuda")
    g0 = p.gains()
    torch.cuda.synchronize()
    p.graph_capture(v, img, gout)
    p.graph_launch()
    p.sync()
    ref, g_ref = img.clone(), gout.clone()
    for T in (41, 700, 701, 3000):
        p.image(_volt(T, T), other)
    p.update()
    p.set_gains(g0)
    p.graph_launch()
    assert p.sync() == 0
    assert _same(img, ref)
    assert torch.max(torch.abs(gout - g_ref)) <= 1e-6 * torch.max(torch.abs(g_ref))     # FP32 sums in another order


def test_pixels_configured_again():
    st = torch.cuda.Stream()
    p = _plan(64, st, path="fused")
    p.configure_pixels([[0.0, 0.0], [0.17, -0.11]])
    v = _volt(40, 1)
    img = torch.zeros((C, 64, 64), dtype=torch.float64, device="cuda")
    g0 = p.gains()
    torch.cuda.synchronize()
    p.graph_capture(v, img)
    p.graph_launch()
    p.sync()
    ref = img.clone()
    p.configure_pixels([[0.0, 0.0], [0.17, -0.11], [0.3, 0.1]])
    p.set_gains(g0)
    p.graph_launch()
    assert p.sync() == 0
    assert _same(img, ref)


def test_callers_capture_of_the_xengine():
    st = torch.cuda.Stream()
    p = _plan(64, st)
    v, longer = _volt(64, 1), _volt(640, 2)
    vis, other = (torch.zeros((C, NA, NA), dtype=torch.complex128, device="cuda") for _ in range(2))
    torch.cuda.synchronize()
    p.visibilities(v, vis)
    p.sync()
    ref = vis.clone()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=st):
        p.visibilities(v, vis)
    p.visibilities(longer, other)
    p.sync()
    vis.zero_()
    torch.cuda.synchronize()
    with torch.cuda.stream(st):
        graph.replay()
    assert p.sync() == 0
    assert torch.equal(vis, ref)
