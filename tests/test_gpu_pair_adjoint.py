"""Frame-pair adjoint (FP32, N = 16..128) against the oracle's analytic
gradient at the edges of its tiles: one to five blocks of 16 in a window,
footprints off 4 and 8, sample counts around a pair and a run, antenna counts
above the CTA size, kernel supports 1, 3 and 5, both voltage formats, a
flagged antenna.  Gradient relative L2 <= 1e-4."""
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


@pytest.mark.parametrize("n,na,rows,cols,T,fmt,support", [
    (16, 6, 9, 14, 3, "c64", 1), (16, 40, 16, 7, 2, "ci4", 3), (32, 70, 29, 17, 9, "ci4", 3),
    (64, 30, 50, 33, 1, "c64", 5), (64, 300, 18, 61, 300, "ci4", 3), (128, 40, 51, 57, 5, "ci4", 3),
    (128, 600, 65, 40, 2, "c64", 3), (128, 25, 13, 68, 4, "c64", 5),
])
def test_pair_adjoint(n, na, rows, cols, T, fmt, support):
    from paper_1603_02126_gb300 import Plan
    rng = np.random.default_rng(3000 + n + na)
    cell_m = 0.5 * 299792458.0 / 50e6
    hx, hy = (((v - support) / 2 - 0.02) * cell_m for v in (cols, rows))
    ant = rng.uniform(-1.0, 1.0, (na, 2)) * [hx, hy]
    ant[0], ant[1] = (-hx, -hy), (hx, hy)
    freqs = [50e6, 46.1e6]
    flags = np.zeros(na, bool)
    flags[2] = True
    sky = np.array([[0.0, 0.0, 4.0], [0.2, -0.15, 1.5]])
    g_true = synth.true_gains(2, na, rng)
    E = synth.voltages(ant, freqs, g_true, sky, T, 0.3, rng)
    lsb = None
    if fmt == "ci4":
        lsb = np.array([0.7, 0.9], np.float32)
        b = synth.quantise_ci4(E, lsb)
        E = O.unpack_ci4(b) * lsb[None, :, None].astype(float)
        dev = torch.from_numpy(b).cuda()
    else:
        dev = torch.from_numpy(E.astype(np.complex64)).cuda()
        E = E.astype(np.complex64).astype(np.complex128)
    g = g_true * (1 + 0.15 * (rng.normal(size=g_true.shape) + 1j * rng.normal(size=g_true.shape)))
    oplan = O.Plan(ant, freqs, n, 0.5, support=support, flags=flags)
    M = O.model_image(oplan, sky)
    ref = O.chi2_gradient(oplan, E, g, M)
    p = Plan(ant, freqs, n, 0.5, support=support, input=fmt, voltage_scale=lsb, flags=flags)
    p.set_gains(g)
    img = p.image(dev)
    dl = 2 * (img - torch.from_numpy(M).cuda())
    grad = p.image_backward(dev, dl).cpu().numpy()
    assert np.linalg.norm(grad - ref) / np.linalg.norm(ref) <= 1e-4
    assert np.all(grad[:, 2] == 0)


@pytest.mark.parametrize("n,na,T", [(32, 40, 5), (64, 300, 33), (128, 60, 4)])
def test_image_of_bf16_gradient_plan(n, na, T):
    """Images and gains of a plan whose gradients are BF16 (the one-frame
    kernel), and of the same plan set back to FP32.  Relative L2 <= 1e-5,
    gains <= 1e-4."""
    from paper_1603_02126_gb300 import Plan
    rng = np.random.default_rng(70 + n)
    half = 7 * 299792458.0 / 50e6
    ant = rng.uniform(-half, half, (na, 2))
    freqs = [50e6, 46.1e6]
    sky = np.array([[0.0, 0.0, 4.0], [0.2, -0.15, 1.5]])
    g0 = synth.true_gains(2, na, rng)
    E = synth.voltages(ant, freqs, g0, sky, T, 0.3, rng).astype(np.complex64)
    oplan = O.Plan(ant, freqs, n, 0.5, support=3, model_lmS=sky)
    g_ref, _, _, ref, _ = O.epical_interval(oplan, E.astype(np.complex128), g0, 0.5)
    dev = torch.from_numpy(E).cuda()
    p = Plan(ant, freqs, n, 0.5, support=3, input="c64")
    for precision in ("bf16", "fp32"):
        p.set_adjoint_precision(precision)
        p.configure((0.0, 0.0), sky, 0.5, g0=g0)
        img = p.image(dev).cpu().numpy()
        p.update()
        assert np.linalg.norm(img - ref) / np.linalg.norm(ref) <= 1e-5
        assert np.max(np.abs(p.gains() - g_ref) / np.abs(g_ref)) <= 1e-4
