"""How long the FP32 partial sums are: one sample 2^14 times as strong as the
others swallows, in an FP32 running sum of |E|^2, every other sample of its
run (each below half a unit in the last place), so the image and the powers
P_a show the runs' length.  At 128 samples at most 16 frame pairs (N = 128) or
32 (N = 512) per partial image, 8 pairs or 8 samples per partial correlation;
the rest must be there to the last sample.  With longer runs short calls were
less accurate than one frame per FP32 value."""
import struct

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


@pytest.mark.parametrize("n,C,half,image_pairs,corr_samples", [(128, 64, 60.0, 16, 16), (512, 8, 250.0, 32, 8)])
def test_runs(n, C, half, image_pairs, corr_samples):
    from paper_1603_02126_gb300 import Plan
    na, T = 5, 128
    ant = np.array([[-half, -half], [half, half], [0.0, 3.0], [-half / 3, half / 2], [half / 2, -1.0]])
    p = Plan(ant, np.linspace(50e6, 48e6, C), n, 0.5, input="c64")
    p.configure((0.0, 0.0), np.array([[0.0, 0.0, 1.0]]), 0.5)
    one = torch.zeros((4, C, na), dtype=torch.complex64, device="cuda")
    one[0] = 1.0
    unit = p.image(one) * 4
    p.update()
    p.configure((0.0, 0.0), np.array([[0.0, 0.0, 1.0]]), 0.5)
    big = float(2 ** 28)
    v = torch.ones((T, C, na), dtype=torch.complex64, device="cuda")
    v[0] = 2.0 ** 14
    v[1] = 0.0                                                # its pair's sum of squares rounds as `unit` does
    img = p.image(v) * T
    bright = unit > 1e-3 * unit.amax(dim=(1, 2), keepdim=True)
    others = (img / unit - big)[bright]                       # samples beside the strong one, of 126
    assert others.max().item() <= 126.5
    assert others.min().item() >= 126 - 2 * (image_pairs - 1) - 0.5
    state = p.get_state()
    head = struct.calcsize("8s6id2q")
    power = np.frombuffer(state, np.float64, C * na, head + 32 * C * na)
    assert power.max() - big <= 126.5
    assert power.min() - big >= 126 - (corr_samples - 2) - 0.5
