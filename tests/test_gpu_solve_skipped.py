"""Pairs that the gain solve leaves out pass nothing on: an antenna all of
whose baselines lie below the cut keeps its start value, also one that is not a
number, and the others solve as if it were flagged (the FP64 oracle, gains to
1e-5: the solve's FP32 pair products).  Channels with one and with several
CTAs."""
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


@pytest.mark.parametrize("value", [np.nan, complex(0.0, np.nan)])
@pytest.mark.parametrize("C,na,scale", [(1, 70, 1.0), (160, 21, 1.0), (2, 70, 2.0 ** 60)])
def test_isolated_antenna(C, na, scale, value):
    from paper_1603_02126_gb300 import Plan
    rng = np.random.default_rng(C + na)
    lam = 299792458.0 / 50e6
    th = np.arange(na) * 2 * np.pi / (na - 1)
    ant = np.stack([2.4 * lam * np.cos(th), 2.4 * lam * np.sin(th)], -1)     # a ring and its centre
    ant[na - 1] = 0.0
    cut = 2.5                                     # wavelengths: every baseline of the centre, some of the ring
    freqs = np.full(C, 50e6)
    sky = np.array([[0.0, 0.0, 5.0], [0.2, 0.1, 1.0], [-0.3, 0.2, 0.7]])
    g = synth.true_gains(C, na, rng)
    VM = np.stack([O.model_visibilities(ant, f, sky) for f in freqs])
    V = g[:, :, None] * np.conj(g[:, None, :]) * VM
    g0 = g * (1 + 0.1 * rng.normal(size=g.shape))
    start = g0 * scale
    start[:, na - 1] = value
    p = Plan(ant, freqs, 64, 0.5, input="c64")
    p.configure((0.0, 0.0), sky, 0.5)
    gd = torch.from_numpy(start).cuda()
    it = p.visibility_solve(torch.from_numpy(V * scale ** 2).cuda(), gd, max_iter=2000, min_baseline=cut)
    gd = gd.cpu().numpy()
    assert (it > 1).all() and (it < 2000).all()
    flags = np.zeros(na, bool)
    flags[na - 1] = True
    far = np.linalg.norm(ant[:, None] - ant[None], axis=-1) / lam >= cut
    for c in {0, C // 2, C - 1}:
        go = O.visibility_solve(V[c], VM[c], g0[c], flags=flags, pair_mask=far)
        assert np.max(np.abs(gd[c, :-1] / scale - go[:-1]) / np.abs(go[:-1])) < 1e-5
        assert np.array_equal(gd[c, -1:], start[c, -1:], equal_nan=True)
