"""epic_plan_set_adjoint_precision is a host call: it allocates nothing and
may be made while a capture is open; the calls after it take BF16 gradients."""
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


@pytest.mark.parametrize("n,half", [(32, 6.0), (64, 40.0), (128, 45.0)])
def test_set_inside_a_capture(n, half):
    from paper_1603_02126_gb300 import Plan
    rng = np.random.default_rng(n)
    na, T = 40, 33
    ant = rng.uniform(-half, half, (na, 2))
    freqs = np.array([50e6, 49e6])
    v = torch.from_numpy(rng.integers(0, 256, (T, 2, na), dtype=np.uint8)).cuda()
    r = torch.randn((2, n, n), dtype=torch.float64, generator=torch.Generator().manual_seed(1)).cuda()
    img, ref = (torch.zeros((2, n, n), dtype=torch.float64, device="cuda") for _ in range(2))
    grad, gref = (torch.zeros((2, na), dtype=torch.complex128, device="cuda") for _ in range(2))
    st = torch.cuda.Stream()
    p, q = (Plan(ant, freqs, n, 0.5, path="fused", stream=st.cuda_stream) for _ in range(2))
    torch.cuda.synchronize()
    q.set_adjoint_precision("bf16")
    q.image(v, ref)
    q.image_backward(v, r, gref)
    p.image_backward(v, r, grad)                 # FP32; the accumulator of the first call
    assert p.sync() == 0 and q.sync() == 0
    free = torch.cuda.mem_get_info()[0]
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=st):
        p.set_adjoint_precision("bf16")
        p.image(v, img)
        p.image_backward(v, r, grad)
    assert torch.cuda.mem_get_info()[0] >= free - (64 << 20)      # the graph's own memory
    graph.replay()
    torch.cuda.synchronize()
    # the same kernels on the same inputs; FP64 sums in another order
    assert torch.linalg.norm(img - ref) <= 1e-12 * torch.linalg.norm(ref)
    assert torch.linalg.norm(grad - gref) <= 1e-12 * torch.linalg.norm(gref)
