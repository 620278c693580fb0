"""Reduced-precision gridding at the edges of its tiles against the FP64
oracle: sample counts around a frame pair, footprints off the row blocks and
with few or many columns, more than one antenna per thread, dense cells whose
lists go through L1, flagged antennas holding NaN, both formats of voltages
and of the transform.  Image relative L2 <= 3e-3, gains <= 1e-4."""
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


@pytest.mark.parametrize("n,na,rows,cols,T,fmt,support,prec,l0", [
    (128, 40, 17, 33, 1, "ci4", 3, "fp16", 0.0), (128, 300, 15, 100, 131, "c64", 5, "bf16", 0.0),
    (256, 700, 109, 60, 5, "ci4", 3, "fp16", 0.08), (256, 90, 8, 200, 4, "c64", 1, "bf16", 0.0),
    (128, 450, 20, 20, 3, "c64", 7, "fp16", 0.0),
])
def test_reduced_precision_interval(n, na, rows, cols, T, fmt, support, prec, l0):
    from paper_1603_02126_gb300 import Plan
    rng = np.random.default_rng(2000 + n + na)
    cell_m = 0.5 * 299792458.0 / 50e6
    hx, hy = (((v - support) / 2 - 0.02) * cell_m for v in (cols, rows))
    ant = rng.uniform(-1.0, 1.0, (na, 2)) * [hx, hy]
    ant[0], ant[1] = (-hx, -hy), (hx, hy)
    freqs = [50e6, 46.1e6]
    flags = np.zeros(na, bool)
    flags[7] = True
    sky = np.array([[l0, 0.0, 5.0], [0.17, -0.11, 1.0]])
    E = synth.voltages(ant, freqs, synth.true_gains(2, na, rng), sky, T, 1.0, rng)
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
    p = Plan(ant, freqs, n, 0.5, support=support, input=fmt, voltage_scale=lsb, flags=flags, precision=prec)
    g0 = synth.true_gains(2, na, rng)
    kw = {}
    if l0:
        p.set_phase_centre(l0, 0.0)
        kw = dict(phase_lm=(l0, 0.0), cal_lm=(l0, 0.0))
    p.configure((l0, 0.0), sky, 0.5, g0=g0)
    img = p.image(dev).cpu().numpy()
    p.update()
    assert p.sync() == 0
    oplan = O.Plan(ant, freqs, n, 0.5, support=support, flags=flags, model_lmS=sky, **kw)
    g_ref, _, _, ref, _ = O.epical_interval(oplan, E, g0, 0.5)
    assert np.linalg.norm(img - ref) / np.linalg.norm(ref) <= 3e-3
    ok = ~flags
    assert np.max(np.abs(p.gains() - g_ref)[:, ok] / np.abs(g_ref)[:, ok]) <= 1e-4
