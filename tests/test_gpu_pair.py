"""Frame-pair imaging (N = 16..128) against the FP64 oracle at the edges of
its tiles: sample counts around a pair, a CTA's share and a partial-image
run; footprints around the 4- and 16-entry blocks of a transform; antenna
counts around the CTA size; both voltage formats; two plans of different
footprints alive at once.  Image relative L2 <= 1e-5, gains <= 1e-4."""
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


def _interval(n, na, span, T, fmt, support, seed):
    """One calibrated interval on an array whose first channel's window has
    `span` rows and columns; returns (plan, voltages, reference image and gains)."""
    from paper_1603_02126_gb300 import Plan
    rng = np.random.default_rng(seed)
    cell_m = 0.5 * 299792458.0 / 50e6
    half = ((span - support) / 2 - 0.02) * cell_m
    ant = rng.uniform(-half, half, (na, 2))
    ant[0], ant[1 % na] = (-half, -half), (half, half)
    freqs = [50e6, 47.3e6]
    sky = np.array([[0.0, 0.0, 5.0], [0.21, -0.13, 1.0]])
    g = synth.true_gains(2, na, rng)
    E = synth.voltages(ant, freqs, g, sky, T, 1.0, rng)
    lsb = None
    if fmt == "ci4":
        lsb = np.array([0.9, 1.1], np.float32)
        b = synth.quantise_ci4(E, lsb)
        E = O.unpack_ci4(b) * lsb[None, :, None].astype(float)
        dev = torch.from_numpy(b).cuda()
    else:
        E = E.astype(np.complex64).astype(np.complex128)
        dev = torch.from_numpy(E.astype(np.complex64)).cuda()
    p = Plan(ant, freqs, n, 0.5, support=support, input=fmt, voltage_scale=lsb)
    g0 = synth.true_gains(2, na, rng)
    p.configure((0.0, 0.0), sky, 0.5, g0=g0)
    oplan = O.Plan(ant, freqs, n, 0.5, support=support, model_lmS=sky)
    g_ref, _, _, ref, _ = O.epical_interval(oplan, E, g0, 0.5)
    return p, dev, ref, g_ref


@pytest.mark.parametrize("n,na,span,T,fmt,support", [
    (16, 5, 9, 1, "c64", 1), (16, 33, 16, 2, "ci4", 3),
    (32, 64, 17, 37, "c64", 3), (32, 65, 30, 301, "ci4", 5),
    (64, 256, 33, 3, "c64", 3), (64, 257, 48, 64, "ci4", 3),
    (128, 512, 49, 40, "ci4", 3), (128, 513, 65, 7, "c64", 5), (128, 30, 16, 700, "ci4", 1),
])
def test_pair_interval(n, na, span, T, fmt, support):
    p, dev, ref, g_ref = _interval(n, na, span, T, fmt, support, 900 + n + na)
    img = p.image(dev).cpu().numpy()
    p.update()
    assert np.linalg.norm(img - ref) / np.linalg.norm(ref) <= 1e-5
    assert np.max(np.abs(p.gains() - g_ref) / np.abs(g_ref)) <= 1e-4


def test_plans_of_different_footprints():
    """A plan keeps working after a smaller one is created."""
    a = _interval(128, 60, 61, 10, "ci4", 3, 1)
    b = _interval(128, 60, 20, 10, "ci4", 3, 2)
    for p, dev, ref, _ in (a, b, a):
        img = p.image(dev).cpu().numpy()
        assert np.linalg.norm(img - ref) / np.linalg.norm(ref) <= 1e-5
