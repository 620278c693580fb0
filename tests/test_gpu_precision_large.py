"""Reduced precision on arrays around the largest whose E' of a frame pair
fits shared memory and well above it, against the FP64 oracle on random
voltages: both voltage formats and transform types, odd sample counts,
flagged antennas holding NaN.  Image relative L2 <= 3e-3, gains <= 1e-4 (the
bounds of the reduced-precision form)."""
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


def _denominators(oplan, sky):
    """D_a of Eq. 16 by sources: sum_s S_s e_a(s) sum_{b != a} conj(A_b e_b(s)),
    without the Na x Na model visibilities."""
    D = []
    for c, f in enumerate(oplan.freqs):
        e = np.exp(-2j * np.pi * (O.antenna_uv(oplan.ant, f) @ sky[:, :2].T))
        A = np.where(oplan.flags, 0.0, oplan.A0[c])
        D.append((e * sky[:, 2]) @ (np.conj(e).T @ np.conj(A)) - np.conj(A) * sky[:, 2].sum())
    return np.stack(D)


@pytest.mark.parametrize("n,na,rows,cols,T,fmt,prec", [
    (128, 13000, 90, 101, 3, "ci4", "fp16"), (128, 14900, 90, 101, 3, "c64", "bf16"),
    (256, 14200, 109, 60, 5, "ci4", "bf16"), (256, 28900, 119, 200, 2, "c64", "fp16"),
])
def test_interval(n, na, rows, cols, T, fmt, prec):
    from paper_1603_02126_gb300 import Plan
    rng = np.random.default_rng(na)
    cell_m = 0.5 * 299792458.0 / 50e6
    hx, hy = (((v - 3) / 2 - 0.02) * cell_m for v in (cols, rows))
    ant = rng.uniform(-1.0, 1.0, (na, 2)) * [hx, hy]
    ant[0], ant[1] = (-hx, -hy), (hx, hy)
    freqs = [50e6, 46.1e6]
    flags = np.zeros(na, bool)
    flags[7] = True
    sky = np.array([[0.0, 0.0, 5.0], [0.17, -0.11, 1.0]])
    g0 = synth.true_gains(2, na, rng)
    E = synth.voltages(ant, freqs, g0, sky, T, 1.0, rng)
    lsb = None
    if fmt == "ci4":
        lsb = np.array([0.9, 1.1], np.float32)
        b = synth.quantise_ci4(E, lsb)
        E = O.unpack_ci4(b) * lsb[None, :, None].astype(float)
        dev = torch.from_numpy(b).cuda()
    else:
        E = E.astype(np.complex64)
        dev = torch.from_numpy(E.copy())
        dev[:, :, 7] = float("nan")
        dev = dev.cuda()
        E = E.astype(np.complex128)
    p = Plan(ant, freqs, n, 0.5, input=fmt, voltage_scale=lsb, flags=flags, precision=prec)
    p.configure((0.0, 0.0), sky, 0.5, g0=g0)
    img = p.image(dev).cpu().numpy()
    p.update()
    p.sync()
    oplan = O.Plan(ant, freqs, n, 0.5, flags=flags)
    oplan.D = _denominators(oplan, sky)
    g_ref, _, _, ref, _ = O.epical_interval(oplan, E, g0, 0.5)
    assert np.linalg.norm(img - ref) / np.linalg.norm(ref) <= 3e-3
    # of the two parts of the update: their sum comes near 0 for one of so many
    assert np.max((np.abs(p.gains() - g_ref) / (np.abs(g_ref) + np.abs(g0)))[:, ~flags]) <= 1e-4
