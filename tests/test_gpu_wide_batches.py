"""Wide frame-pair form over calls of several large batches (hundreds of
samples each, more than one FP32 run of pairs), against the FP64 oracle: a
scratch budget whose share per sample of all channels is an odd number just
above 256, sample counts around one and two batches, both voltage formats.
Image relative L2 <= 1e-5, gains <= 1e-4 (the bounds of the plain path)."""
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


def _stride(rows):
    while rows % 16 != 4:
        rows += 1
    return rows


@pytest.mark.parametrize("n,na,rows,T,C,fmt,quotient", [
    (128, 200, 100, 256, 2, "ci4", 257), (128, 200, 100, 257, 3, "c64", 257), (128, 90, 97, 515, 2, "ci4", 301),
    (256, 60, 33, 258, 2, "c64", 257), (256, 60, 100, 515, 3, "ci4", 257), (256, 40, 17, 603, 2, "c64", 301),
])
def test_large_batches(n, na, rows, T, C, fmt, quotient):
    from paper_1603_02126_gb300 import Plan
    rng = np.random.default_rng(4000 + n + T)
    cell_m = 0.5 * 299792458.0 / 50e6
    h = ((rows - 3) / 2 - 0.02) * cell_m
    ant = rng.uniform(-h, h, (na, 2))
    ant[0], ant[1] = (-h, -h), (h, h)
    freqs = np.linspace(50e6, 45e6, C)
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
    kw = dict(input=fmt, voltage_scale=lsb, path="fused" if n == 128 else "unfused")
    probe = Plan(ant, freqs, n, 0.5, **kw)
    budget = quotient * C * n * _stride(probe.info()["window_rows"]) * 8 + 1000
    probe.close()
    p = Plan(ant, freqs, n, 0.5, workspace_bytes=budget, **kw)
    g0 = synth.true_gains(C, na, rng)
    p.configure((0.0, 0.0), sky, 0.5, g0=g0)
    img = p.image(dev).cpu().numpy()
    p.update()
    assert p.sync() == 0
    oplan = O.Plan(ant, freqs, n, 0.5, model_lmS=sky)
    g_ref, _, _, ref, _ = O.epical_interval(oplan, E, g0, 0.5)
    assert np.linalg.norm(img - ref) / np.linalg.norm(ref) <= 1e-5
    assert np.max(np.abs(p.gains() - g_ref) / np.abs(g_ref)) <= 1e-4
