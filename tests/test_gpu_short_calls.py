"""Calls of one to four samples, where the plan chooses between the one-frame
and the frame-pair kernels and gives each CTA one pair, and footprints on
both sides of the line between the one-frame kernel and the wide form
(N = 128), against the FP64 oracle: image relative L2 <= 1e-5, gains and
gradient <= 1e-4 (the bounds of the plain path)."""
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


def _setup(n, na, rows, T, C, fmt):
    from paper_1603_02126_gb300 import Plan
    rng = np.random.default_rng(6000 + n + na + T)
    cell_m = 0.5 * 299792458.0 / 50e6
    h = ((rows - 3) / 2 - 0.02) * cell_m
    ant = rng.uniform(-h, h, (na, 2))
    ant[0], ant[1] = (-h, -h), (h, h)
    freqs = np.linspace(50e6, 40e6, C)
    sky = np.array([[0.0, 0.0, 5.0], [0.21, -0.13, 1.0]])
    g0 = synth.true_gains(C, na, rng)
    E = synth.voltages(ant, freqs, g0, sky, T, 1.0, rng)
    lsb = None
    if fmt == "ci4":
        lsb = np.linspace(0.9, 1.1, C).astype(np.float32)
        b = synth.quantise_ci4(E, lsb)
        E = O.unpack_ci4(b) * lsb[None, :, None].astype(float)
        dev = torch.from_numpy(b).cuda()
    else:
        dev = torch.from_numpy(E.astype(np.complex64)).cuda()
        E = E.astype(np.complex64).astype(np.complex128)
    p = Plan(ant, freqs, n, 0.5, input=fmt, voltage_scale=lsb, path="fused")
    return p, dev, E, g0, sky, O.Plan(ant, freqs, n, 0.5, model_lmS=sky)


@pytest.mark.parametrize("T", [1, 2, 3, 4])
@pytest.mark.parametrize("n,na,rows,C,fmt", [
    (16, 12, 9, 1, "c64"), (32, 100, 25, 40, "ci4"), (64, 60, 51, 33, "c64"), (128, 100, 51, 20, "ci4"),
    (128, 60, 97, 20, "c64"),
])
def test_interval(n, na, rows, T, C, fmt):
    p, dev, E, g0, sky, oplan = _setup(n, na, rows, T, C, fmt)
    p.configure((0.0, 0.0), sky, 0.5, g0=g0)
    img = p.image(dev).cpu().numpy()
    p.update()
    assert p.sync() == 0
    g_ref, _, _, ref, _ = O.epical_interval(oplan, E, g0, 0.5)
    assert np.linalg.norm(img - ref) / np.linalg.norm(ref) <= 1e-5
    assert np.max(np.abs(p.gains() - g_ref) / np.abs(g_ref)) <= 1e-4


@pytest.mark.parametrize("T", [1, 2])
@pytest.mark.parametrize("n,na,rows,C,fmt", [(16, 12, 9, 2, "c64"), (64, 60, 51, 3, "ci4"), (128, 100, 51, 2, "c64")])
def test_gradient(n, na, rows, T, C, fmt):
    p, dev, E, g0, sky, oplan = _setup(n, na, rows, T, C, fmt)
    g = g0 * 1.1
    M = O.model_image(oplan, sky)
    p.set_gains(g)
    dl = 2 * (p.image(dev) - torch.from_numpy(M).cuda())
    grad = p.image_backward(dev, dl).cpu().numpy()
    ref = O.chi2_gradient(oplan, E, g, M)
    assert np.linalg.norm(grad - ref) / np.linalg.norm(ref) <= 1e-4


@pytest.mark.parametrize("na,rows,wide", [(100, 107, True), (100, 109, False), (250, 113, True), (700, 113, False)])
def test_form_by_footprint(na, rows, wide):
    p, dev, E, g0, sky, oplan = _setup(128, na, rows, 5, 2, "ci4")
    p.configure((0.0, 0.0), sky, 0.5, g0=g0)
    img = p.image(dev).cpu().numpy()
    assert (p.info()["batch_time"] > 0) == wide
    p.update()
    g_ref, _, _, ref, _ = O.epical_interval(oplan, E, g0, 0.5)
    assert np.linalg.norm(img - ref) / np.linalg.norm(ref) <= 1e-5
    assert np.max(np.abs(p.gains() - g_ref) / np.abs(g_ref)) <= 1e-4
