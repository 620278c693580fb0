"""The gain solve does not depend on the units: fluxes and gains scaled by
powers of two (a model in SI units is near 1e-26) give the same solution,
scaled, as long as the visibilities themselves are FP32 numbers.  Each solve agrees with an FP64 solve to about 1e-6 (its FP32 pair
products), so two agree to 4e-6."""
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


def _problem(C, na):
    rng = np.random.default_rng(C + na)
    ant = synth.layout_disc(na, 22.0, rng)
    freqs = np.linspace(48e6, 62e6, C)
    sky = np.array([[0.0, 0.0, 5.0], [0.2, 0.1, 1.0], [-0.3, 0.2, 0.7]])
    g = synth.true_gains(C, na, rng)
    V = np.stack([O.model_visibilities(ant, f, sky) for f in freqs]) * g[:, :, None] * np.conj(g[:, None, :])
    return ant, freqs, sky, g, V, g * (1 + 0.1 * rng.normal(size=g.shape))


def _solve(ant, freqs, sky, V, g0, **kw):
    from paper_1603_02126_gb300 import Plan
    p = Plan(ant, freqs, 64, 0.5, input="c64")
    p.configure((0.0, 0.0), sky, 0.5)
    gd = torch.from_numpy(g0.astype(np.complex128)).cuda()
    it = p.visibility_solve(torch.from_numpy(V).cuda(), gd, max_iter=2000, **kw)
    return gd.cpu().numpy(), it


@pytest.mark.parametrize("C,na", [(1, 130), (20, 33)])
@pytest.mark.parametrize("flux,gain", [(-86, 40), (-86, 0), (70, -32), (-100, 70), (0, 60), (0, -60)])
def test_units(C, na, flux, gain):
    ant, freqs, sky, g, V, g0 = _problem(C, na)
    ref, it_ref = _solve(ant, freqs, sky, V, g0)
    sky2 = sky * [1.0, 1.0, 2.0 ** flux]
    got, it = _solve(ant, freqs, sky2, V * 2.0 ** (flux + 2 * gain), g0 * 2.0 ** gain)
    assert (it > 1).all() and (np.abs(it - it_ref) <= 1).all()
    assert np.max(np.abs(got / 2.0 ** gain - ref) / np.abs(ref)) <= 4e-6


def test_start_far_from_the_solution():
    ant, freqs, sky, g, V, g0 = _problem(2, 40)
    scale = 2.0 ** 40
    sky2 = sky * [1.0, 1.0, 2.0 ** -86]
    got, it = _solve(ant, freqs, sky2, V * 2.0 ** (2 * 40 - 86), np.ones_like(g0))
    ref, _ = _solve(ant, freqs, sky, V, np.ones_like(g0) / scale)
    assert (it < 2000).all()
    assert np.max(np.abs(got / scale - ref) / np.abs(ref)) <= 4e-6
