"""Frame-pair form through HBM (N = 256, 512, and N = 128 with a footprint
too large for one SM) against the FP64 oracle at
the edges of its tiles: sample counts around a pair and a batch, footprints
around the 4-row, row-block and 32-entry edges, one channel and several,
scratch budgets of one pair and of part of the channels, both voltage
formats.  Image relative L2 <= 1e-5, gains <= 1e-4."""
import numpy as np
import pytest

import epic_synth as synth
import oracle as O

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__
    __graft_entry__.build()


@pytest.mark.parametrize("n,na,rows,cols,T,C,fmt,support,budget", [
    (256, 40, 17, 33, 1, 1, "ci4", 3, 0), (256, 300, 96, 129, 5, 3, "c64", 5, 1 << 21),
    (256, 700, 250, 61, 4, 2, "ci4", 3, 1), (256, 90, 32, 32, 260, 1, "c64", 1, 0),
    (512, 60, 8, 40, 3, 2, "ci4", 3, 0), (512, 500, 261, 257, 2, 2, "c64", 3, 3 << 20),
    (512, 200, 505, 500, 2, 1, "ci4", 3, 0), (128, 90, 97, 101, 67, 3, "ci4", 3, 0),
    (128, 200, 127, 90, 9, 2, "c64", 5, 0), (128, 700, 70, 127, 3, 2, "ci4", 3, 1 << 20),
])
def test_wide_interval(n, na, rows, cols, T, C, fmt, support, budget):
    from paper_1603_02126_gb300 import Plan
    rng = np.random.default_rng(1000 + n + na)
    cell_m = 0.5 * 299792458.0 / 50e6
    hx, hy = (((v - support) / 2 - 0.02) * cell_m for v in (cols, rows))
    ant = rng.uniform(-1.0, 1.0, (na, 2)) * [hx, hy]
    ant[0], ant[1] = (-hx, -hy), (hx, hy)
    freqs = np.linspace(50e6, 41e6, C)
    sky = np.array([[0.0, 0.0, 5.0], [0.17, -0.11, 1.0]])
    E = synth.voltages(ant, freqs, synth.true_gains(C, na, rng), sky, T, 1.0, rng)
    lsb = None
    if fmt == "ci4":
        lsb = np.linspace(0.9, 1.1, C).astype(np.float32)
        b = synth.quantise_ci4(E, lsb)
        E = O.unpack_ci4(b) * lsb[None, :, None].astype(float)
        dev = torch.from_numpy(b).cuda()
    else:
        E = E.astype(np.complex64).astype(np.complex128)
        dev = torch.from_numpy(E.astype(np.complex64)).cuda()
    p = Plan(ant, freqs, n, 0.5, support=support, input=fmt, voltage_scale=lsb,
             path="fused" if n == 128 else "unfused", workspace_bytes=budget)
    g0 = synth.true_gains(C, na, rng)
    p.configure((0.0, 0.0), sky, 0.5, g0=g0)
    img = p.image(dev).cpu().numpy()
    p.update()
    assert p.sync() == 0
    oplan = O.Plan(ant, freqs, n, 0.5, support=support, model_lmS=sky)
    g_ref, _, _, ref, _ = O.epical_interval(oplan, E, g0, 0.5)
    assert np.linalg.norm(img - ref) / np.linalg.norm(ref) <= 1e-5
    assert np.max(np.abs(p.gains() - g_ref) / np.abs(g_ref)) <= 1e-4
