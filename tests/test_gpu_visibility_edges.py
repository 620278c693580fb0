"""X-engine packing and the gain solve at the edges of their tiles, against
the FP64 oracle: 4-bit sums exact for antenna counts off the word, block and
tile sizes, sample counts around a block, and an unaligned buffer; solves
with one to eight CTAs per channel, antenna counts off the row groups, and
NaN in a flagged antenna's visibilities (gains to 1e-5, the solve's FP32
pair products)."""
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


@pytest.mark.parametrize("na,T,C,shift", [(3, 1, 2, 0), (5, 33, 1, 0), (64, 64, 2, 1), (130, 95, 2, 0), (132, 65, 1, 2)])
def test_xengine_exact(na, T, C, shift):
    from paper_1603_02126_gb300 import Plan
    rng = np.random.default_rng(na + T)
    b = rng.integers(0, 256, (T, C, na), dtype=np.uint8)
    buf = torch.zeros(b.size + shift, dtype=torch.uint8, device="cuda")
    d = buf[shift:].view(T, C, na)
    d.copy_(torch.from_numpy(b))
    ant = synth.layout_disc(na, 20.0, rng)
    p = Plan(ant, np.linspace(48e6, 50e6, C), 64, 0.5, input="ci4")
    V = p.visibilities(d).cpu().numpy() * T
    E = O.unpack_ci4(b)
    for c in range(C):
        ref = E[:, c].T @ E[:, c].conj()
        assert np.array_equal(np.rint(V[c].real), ref.real) and np.array_equal(np.rint(V[c].imag), ref.imag)
        assert np.max(np.abs(V[c] - ref)) <= 1e-9 * T


@pytest.mark.parametrize("C,na", [(1, 9), (1, 301), (3, 130), (20, 70), (160, 33)])
def test_solve_cluster_sizes(C, na):
    from paper_1603_02126_gb300 import Plan
    rng = np.random.default_rng(C + na)
    ant = synth.layout_disc(na, 22.0, rng)
    freqs = np.linspace(48e6, 62e6, C)
    flags = np.zeros(na, bool)
    flags[na // 2] = True
    sky = np.array([[0.0, 0.0, 5.0], [0.2, 0.1, 1.0], [-0.3, 0.2, 0.7]])
    g = synth.true_gains(C, na, rng)
    VM = np.stack([O.model_visibilities(ant, f, sky) for f in freqs])
    noise = 0.05 * (rng.normal(size=VM.shape) + 1j * rng.normal(size=VM.shape))
    V = g[:, :, None] * np.conj(g[:, None, :]) * VM + noise + np.conj(np.swapaxes(noise, 1, 2))
    g0 = g * (1 + 0.1 * rng.normal(size=g.shape))
    Vd = V.copy()
    Vd[:, na // 2, :] = np.nan
    Vd[:, :, na // 2] = np.nan
    p = Plan(ant, freqs, 64, 0.5, input="c64", flags=flags)
    p.configure((0.0, 0.0), sky, 0.5)
    gd = torch.from_numpy(g0).cuda()
    it = p.visibility_solve(torch.from_numpy(Vd).cuda(), gd, max_iter=2000)
    gd = gd.cpu().numpy()
    assert (it > 1).all() and (it < 2000).all()
    for c in {0, C // 2, C - 1}:
        go = O.visibility_solve(V[c], VM[c], g0[c], flags=flags)
        assert np.max(np.abs(gd[c] - go) / np.abs(go)) < 1e-5
        assert gd[c, na // 2] == g0[c, na // 2]
