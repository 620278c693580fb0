"""The work this framework is used for, as cases to time and compare.

A case is one call of a user's program through the public entry points: a
calibration interval (image + EPICal update) of an array on the device or
from host buffers, a reduced-precision interval, one gradient of the
image-versus-model chi-squared, or the visibility comparison (X-engine and
StEFCal solve).  The sizes are those of the repository's workloads and
benchmark, and generic ones between them.

Images and gains leave the library as float64 accumulators of FP32 (or
reduced-precision) arithmetic; a program that keeps them stores them in
single precision, which is what `run` returns.  Visibilities of 4-bit
voltages are exact sums and stay complex128.
"""
from __future__ import annotations

import math

import numpy as np
import torch

C_LIGHT = 299792458.0
CELL = 0.5                      # grid cell, wavelengths
SIGMA = 0.5                     # Gaussian illumination kernel, cells


def _case(**kw):
    c = dict(kind="interval", layout="ellipse", n_ant=256, semi_x=50.0, semi_y=45.0, pitch=0.0, f_lo=40e6,
             f_hi=80e6, n_chan=64, n_time=1024, grid_n=128, input="ci4", support=3, precision="fp32",
             gamma=0.5, n_src=50, n_flag=0, phase_l=0.0, phase_m=0.0)
    c.update(kw)
    return c


def listed():
    return [
        # the smallest interval: a 32-antenna array, one channel, complex64;
        # launches and latency count
        _case(name="tiny_interval", n_ant=32, semi_x=10.0, semi_y=10.0, f_lo=50e6, f_hi=50e6, n_chan=1,
              n_time=2000, grid_n=32, input="c64", n_src=4),
        # a station on a 64 x 64 grid: odd counts, complex64 voltages, a 5 x 5
        # kernel, flagged antennas, phased off zenith
        _case(name="station64_c64", n_ant=248, n_chan=15, n_time=1023, grid_n=64, input="c64", support=5,
              n_flag=9, phase_l=0.11, phase_m=-0.07),
        # the station interval of the benchmark: 256 antennas, 64 channels,
        # 128 x 128, 10^4 4-bit samples
        _case(name="lwa_interval", n_time=10000),
        # the same station with the shortest calibration interval of the
        # noise-trend study: 128 samples
        _case(name="lwa_short", n_time=128, gamma=0.35),
        # the same through host buffers (upload, image, download, update):
        # a program that receives its samples in host memory
        _case(name="lwa_host", kind="host", n_time=2048),
        # the station in reduced precision, an odd number of samples
        _case(name="lwa_bf16", n_time=2001, precision="bf16"),
        # 1024 compact antennas, 256 x 256: plain FP32
        _case(name="compact_fp32", n_ant=1024, semi_x=100.0, semi_y=100.0, n_chan=32, n_time=4096, grid_n=256),
        # the same in FP16 on the tensor cores
        _case(name="compact_fp16", n_ant=1024, semi_x=100.0, semi_y=100.0, n_chan=32, n_time=4096, grid_n=256,
              precision="fp16"),
        # 2048 antennas on a jittered hexagonal lattice, 256 channels,
        # 512 x 512, complex64: the largest grid and array
        _case(name="hex_fp32", layout="hex", n_ant=2048, pitch=8.0, f_lo=50e6, f_hi=100e6, n_chan=256, n_time=128,
              grid_n=512, input="c64"),
        # one forward and backward pass of the differentiable image
        _case(name="grad_fp32", kind="grad", n_chan=16, n_time=4096),
        # the same with BF16 transforms in the adjoint, an odd sample count
        _case(name="grad_bf16", kind="grad", n_chan=16, n_time=1023, precision="bf16"),
        # the visibility comparison: X-engine over one effective integration
        # time and the gain solve on its visibilities
        _case(name="visibility_solve", kind="vis", n_time=4254, gamma=0.35),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["interval", "interval", "interval", "host", "precision", "precision", "grad", "vis"])
    n = rng.choice([32, 64, 128, 128, 256, 512])
    if kind == "precision":
        n = rng.choice([128, 256])
    if kind in ("grad", "host"):
        n = rng.choice([32, 64, 128])
    if kind == "vis":
        n = 128
    na = _log(rng, 64 if kind == "vis" else 16, {32: 100, 64: 300, 128: 512, 256: 1024, 512: 2048}[n])
    nc = _log(rng, 1, 64)
    f_lo = rng.uniform(30e6, 80e6)
    f_hi = f_lo * rng.uniform(1.0, 2.0) if nc > 1 else f_lo
    support = rng.choice([1, 3, 3, 3, 5]) if kind != "precision" else 3
    # semi-axes that put the footprint's edge at 40 to 95 per cent of the
    # grid's half side at the highest frequency (at most 128 rows for the
    # reduced-precision form)
    half = (n / 2 - 1 - support) * CELL * C_LIGHT / f_hi
    if kind == "precision":
        half = min(half, (62 - support) * CELL * C_LIGHT / f_hi)
    semi_x, semi_y = half * rng.uniform(0.4, 0.95), half * rng.uniform(0.4, 0.95)
    # at most about half the arithmetic of the largest listed case, or 2 GB of voltages
    frames = 8e10 / (n * n * math.log2(n * n))
    most = min(10000, int(frames / nc), int(2.5e8 / (nc * na)))
    t = _log(rng, 500 if kind == "vis" else 16, min(most, 5000) if kind == "vis" else most)
    c = _case(kind="interval" if kind == "precision" else kind, n_ant=na, n_chan=nc, n_time=t, grid_n=n,
              semi_x=semi_x, semi_y=semi_y, f_lo=f_lo, f_hi=f_hi, support=support,
              input="ci4" if kind == "vis" else rng.choice(["ci4", "ci4", "c64"]),
              gamma=rng.choice([0.35, 0.5, 0.7]), n_src=_log(rng, 3, 50),
              n_flag=rng.choice([0, 0, 1, na // 16]))
    if kind == "precision":
        c["precision"] = rng.choice(["fp16", "bf16"])
    if kind == "grad":
        c["precision"] = rng.choice(["fp32", "fp32", "bf16"])
    return c


# --------------------------------------------------------------------------
# inputs
# --------------------------------------------------------------------------
def _array(case, rng):
    na = case["n_ant"]
    if case["layout"] == "hex":
        r = int(math.ceil(math.sqrt(na))) + 2
        i, j = np.meshgrid(np.arange(-r, r + 1), np.arange(-r, r + 1), indexing="ij")
        pts = np.stack([case["pitch"] * (i + 0.5 * j), case["pitch"] * math.sqrt(0.75) * j], -1).reshape(-1, 2)
        pts = pts[np.argsort(np.hypot(pts[:, 0], pts[:, 1]), kind="stable")[:na]]
        return pts + rng.uniform(-0.5, 0.5, size=pts.shape)
    r = np.sqrt(rng.uniform(0.0, 1.0, na))
    th = rng.uniform(0.0, 2 * np.pi, na)
    return np.stack([case["semi_x"] * r * np.cos(th), case["semi_y"] * r * np.sin(th)], -1)


def _sky(case, rng):
    """Point sources with dN/dS ~ S^-2 on [0.5, 50] at l^2 + m^2 < 0.5; the
    brightest, the calibrator, at the phase centre."""
    n = case["n_src"]
    s = 1.0 / (2.0 - rng.uniform(size=n) * (2.0 - 0.02))
    r, th = np.sqrt(0.5 * rng.uniform(size=n)), rng.uniform(0, 2 * np.pi, n)
    sky = np.stack([r * np.cos(th), r * np.sin(th), s], -1)[np.argsort(-s, kind="stable")]
    sky[0] = (case["phase_l"], case["phase_m"], max(10.0, sky[0, 2]))
    return sky


def _setup(case, seed):
    # the array and its broken antennas are the station's own; sky, gains and
    # voltages come from the seed
    na, nc = case["n_ant"], case["n_chan"]
    station = np.random.default_rng(na)
    ant = _array(case, station)
    flags = np.zeros(na, np.uint8)
    flags[station.choice(na, case["n_flag"], replace=False)] = 1
    rng = np.random.default_rng(seed)
    sky = _sky(case, rng)
    freqs = np.linspace(case["f_lo"], case["f_hi"], nc)
    true = np.abs(rng.normal(1.0, 0.1, (nc, na)).clip(0.3)) * np.exp(1j * rng.uniform(-np.pi, np.pi, (nc, na)))
    # gains in hand: those of an earlier interval, near the true ones
    g0 = true * (1 + 0.05 * (rng.normal(size=(nc, na)) + 1j * rng.normal(size=(nc, na))))
    noise = sky[:, 2].sum() / 5.0
    lsb = np.full(nc, math.sqrt((1.01 * sky[:, 2].sum() + noise) / 2) / 2.0, np.float32)
    return dict(ant=ant, sky=sky, freqs=freqs, true=true, g0=g0, noise=noise, lsb=lsb, flags=flags)


def _voltages(case, s, seed):
    """E_a = g_a sum_s sqrt(S_s) z_s(t) exp(-2 pi i u_a . s_s) + n_a(t) on the
    GPU: complex64, or rounded to 4-bit parts in one byte."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))
    T, nc, na = case["n_time"], case["n_chan"], case["n_ant"]
    out = torch.empty((T, nc, na), dtype=torch.uint8 if case["input"] == "ci4" else torch.complex64, device="cuda")
    amp = torch.as_tensor(np.sqrt(s["sky"][:, 2] / 2), dtype=torch.float32, device="cuda")
    for c, f in enumerate(s["freqs"]):
        u = s["ant"] * f / C_LIGHT
        ph = s["true"][c][:, None] * np.exp(-2j * np.pi * (u @ s["sky"][:, :2].T))
        ph = torch.as_tensor(ph, device="cuda").to(torch.complex64)
        z = torch.view_as_complex(torch.randn((T, len(amp), 2), generator=gen, device="cuda")) * amp
        n = torch.view_as_complex(torch.randn((T, na, 2), generator=gen, device="cuda"))
        e = z @ ph.T + n * math.sqrt(s["noise"] / 2)
        if case["input"] == "ci4":
            q = torch.view_as_real(e).div_(float(s["lsb"][c])).round_().clamp_(-7, 7).to(torch.int32) & 15
            out[:, c] = ((q[..., 0] << 4) | q[..., 1]).to(torch.uint8)
        else:
            out[:, c] = e
    return out


def _model_image(case, s, taps):
    """Image of the sky model with unit gains: sum_s S_s |sum_a A_ka e_a|^2."""
    img = torch.empty((case["n_chan"], case["grid_n"], case["grid_n"]), dtype=torch.float64, device="cuda")
    for c, f in enumerate(s["freqs"]):
        u = s["ant"] * f / C_LIGHT
        e = np.sqrt(s["sky"][:, 2])[:, None] * np.exp(-2j * np.pi * (s["sky"][:, :2] @ u.T))
        x = _fields(case, taps[c], torch.as_tensor(e, device="cuda"))
        img[c] = (x.real ** 2 + x.imag ** 2).sum(0)
    return img


def prepare(case, seed):
    from paper_1603_02126_gb300 import Plan
    s = _setup(case, seed)
    kind = case["kind"]
    plan = Plan(s["ant"], s["freqs"], case["grid_n"], CELL, support=case["support"], param=SIGMA,
                input=case["input"], voltage_scale=s["lsb"] if case["input"] == "ci4" else None,
                flags=s["flags"] if case["n_flag"] else None,
                precision=case["precision"] if kind != "grad" else "fp32")
    volt = _voltages(case, s, seed)
    st = dict(kind=kind, plan=plan, volt=volt)
    nc, na, n = case["n_chan"], case["n_ant"], case["grid_n"]
    if kind == "grad":
        plan.set_adjoint_precision(case["precision"])
        taps = [_taps(case, s, f) for f in s["freqs"]]
        st["model"] = _model_image(case, s, taps)
        st["g"] = torch.as_tensor(s["g0"], device="cuda").requires_grad_(True)
        return st
    if case["phase_l"] or case["phase_m"]:
        plan.set_phase_centre(case["phase_l"], case["phase_m"])
    plan.configure((case["phase_l"], case["phase_m"]), s["sky"], case["gamma"], g0=s["g0"])
    st["gains"] = torch.empty((nc, na), dtype=torch.complex128, device="cuda")
    if kind == "host":
        st["volt"] = volt.cpu().pin_memory()
        st["image"] = torch.empty((nc, n, n), dtype=torch.float64).pin_memory()
    elif kind == "vis":
        st["g0"] = torch.as_tensor(s["g0"], device="cuda")
        st["vis"] = torch.empty((nc, na, na), dtype=torch.complex128, device="cuda")
    else:
        st["image"] = torch.empty((nc, n, n), dtype=torch.float64, device="cuda")
    return st


def run(st):
    plan, kind = st["plan"], st["kind"]
    if kind == "grad":
        from paper_1603_02126_gb300.autograd import EpicImageFn, chi2
        g = st["g"]
        g.grad = None
        image = EpicImageFn.apply(g, st["volt"], plan)
        chi2(image, st["model"]).backward()
        return {"image": image.detach().float(), "grad": g.grad.to(torch.complex64)}
    if kind == "vis":
        plan.visibilities(st["volt"], st["vis"])
        gains = st["g0"].clone()
        plan.visibility_solve(st["vis"], gains)
        return {"vis": st["vis"], "gains": gains.to(torch.complex64)}
    if kind == "host":
        image = plan.image_host(st["volt"], st["image"])
        plan.update(st["gains"])
        return {"image": image.float(), "gains": st["gains"].to(torch.complex64)}
    plan.image(st["volt"], st["image"])
    plan.update(st["gains"])
    return {"image": st["image"].float(), "gains": st["gains"].to(torch.complex64)}


# --------------------------------------------------------------------------
# what a pass cannot do without, and its answer in 64 bits
# --------------------------------------------------------------------------
def work(case):
    T, nc, na, n, k = (case[x] for x in ("n_time", "n_chan", "n_ant", "grid_n", "support"))
    volt = T * nc * na * (1 if case["input"] == "ci4" else 8)
    if case["kind"] == "vis":
        # each distinct pair once; the solve reads V and the model once
        return {"bytes": volt + 3 * nc * na * na * 16 + 2 * nc * na * 16, "flops": 4.0 * T * nc * na * na}
    # gain 6 Na, gridding 4 Na K^2, FFT 5 N^2 log2 N^2, square 3 N^2, correlation 11 Na, per frame
    frame = 6 * na + 4 * na * k * k + 5 * n * n * math.log2(n * n) + 3 * n * n + 11 * na
    out = nc * n * n * 12 + nc * na * 24
    if case["kind"] == "grad":
        # forward image, then recomputed transform, inverse transform, degridding
        frame = 2 * frame + 5 * n * n * math.log2(n * n) + 4 * na * k * k
        return {"bytes": volt + out + 2 * nc * n * n * 8, "flops": float(T) * nc * frame}
    return {"bytes": volt + out, "flops": float(T) * nc * frame}


def _taps(case, s, f):
    """Stencil cells [Na][K^2] (flat grid index) and normalised weights of
    one channel on the GPU; weights of flagged antennas are zero."""
    n, k = case["grid_n"], case["support"]
    p = (s["ant"] * f) / C_LIGHT / CELL + n // 2
    b = np.floor(p + 0.5).astype(np.int64)
    d = np.arange(k) - (k - 1) // 2
    jx, jy = b[:, 0, None] + d, b[:, 1, None] + d
    wx = np.exp(-(jx - p[:, 0, None]) ** 2 / (2 * SIGMA ** 2))
    wy = np.exp(-(jy - p[:, 1, None]) ** 2 / (2 * SIGMA ** 2))
    w = (wy[:, :, None] * wx[:, None, :]).reshape(len(p), -1)
    w = w / w.sum(1, keepdims=True) * (s["flags"] == 0)[:, None]
    idx = np.clip((jy[:, :, None] * n + jx[:, None, :]).reshape(len(p), -1), 0, n * n - 1)
    return torch.as_tensor(idx, device="cuda"), torch.as_tensor(w, device="cuda")


def _fields(case, taps, e):
    """E-field images [t][N][N] (centred) of gain-corrected voltages e [t][Na]."""
    n = case["grid_n"]
    idx, w = taps
    grid = torch.zeros((n * n, e.shape[0]), dtype=torch.complex128, device="cuda")
    et = e.T.contiguous()
    for j in range(idx.shape[1]):
        grid.index_add_(0, idx[:, j], et * w[:, j, None])
    grid = torch.fft.ifftshift(grid.T.reshape(-1, n, n), dim=(1, 2))
    return torch.fft.fftshift(torch.fft.ifft2(grid, norm="forward"), dim=(1, 2)) / case["n_ant"]


def _exact_volt(case, s, volt, c):
    if case["input"] == "c64":
        return volt[:, c].to(torch.complex128)
    b = volt[:, c].to(torch.int32)
    re, im = (b << 24) >> 28, (b << 28) >> 28
    return torch.complex(re.double(), im.double()) * float(s["lsb"][c])


def _phasors(s, f, lm):
    """e^{+2 pi i u_a . s} [Ns][Na] for directions lm [Ns][2]."""
    u = (s["ant"] * f) / C_LIGHT
    return np.exp(2j * np.pi * (np.atleast_2d(lm) @ u.T))


def _exact_gains(case, s, f, c, taps, e, pix):
    """EPICal's damped update (Eqs. 12, 15-17) of one channel, calibrator at
    the phase centre: A_0 = p_a / Na there."""
    na = case["n_ant"]
    live = s["flags"] == 0
    p = _phasors(s, f, [(case["phase_l"], case["phase_m"])])[0]
    a0 = p / na * live
    ph = _phasors(s, f, s["sky"][:, :2])
    b = (np.conj(a0) * ph).sum(1)
    d = ((s["sky"][:, 2] * b)[:, None] * np.conj(ph)).sum(0) - s["sky"][:, 2].sum() * np.conj(a0)
    k = (e * pix.conj()[:, None]).mean(0).cpu().numpy()
    pw = (e.real ** 2 + e.imag ** 2).mean(0).cpu().numpy()
    g = s["g0"][c]
    new = (1 - case["gamma"]) * (k - np.conj(a0) * pw / np.conj(g)) / np.where(live, d, 1) + case["gamma"] * g
    return np.where(live, new, g)


def _exact_solve(case, s, vis):
    """Eq. 21 by StEFCal, every other iterate averaged, to 1e-12."""
    model = []
    for f in s["freqs"]:
        ph = np.conj(_phasors(s, f, s["sky"][:, :2]))
        model.append((ph.T * s["sky"][:, 2]) @ np.conj(ph))
    m = torch.as_tensor(np.stack(model), device="cuda")
    live = torch.as_tensor(s["flags"] == 0, device="cuda")
    off = (live[:, None] & live[None, :] & ~torch.eye(len(live), dtype=torch.bool, device="cuda"))
    m, v = m * off, vis * off
    g = torch.as_tensor(s["g0"], device="cuda")
    for it in range(400):
        z = g[:, None, :] * m.conj()
        den = (z.real ** 2 + z.imag ** 2).sum(2)
        x = torch.where(den > 0, (v * z).sum(2) / den.clamp_min(1e-300), g)
        if it & 1:
            x = 0.5 * (x + g)
        done = ((x - g).abs().amax(1) <= 1e-12 * x.abs().amax(1)).all()
        g = x
        if done:
            break
    return g


def exact(case, seed):
    s = _setup(case, seed)
    volt = _voltages(case, s, seed)
    T, nc, na, n = case["n_time"], case["n_chan"], case["n_ant"], case["grid_n"]
    if case["kind"] == "vis":
        vis = torch.empty((nc, na, na), dtype=torch.complex128, device="cuda")
        for c in range(nc):
            e = _exact_volt(case, s, volt, c)
            vis[c] = e.T @ e.conj() / T
        return {"vis": vis, "gains": _exact_solve(case, s, vis)}
    step = max(1, (1 << 28) // (n * n))
    image = torch.zeros((nc, n, n), dtype=torch.float64, device="cuda")
    taps = [_taps(case, s, f) for f in s["freqs"]]
    gains = np.empty((nc, na), complex)
    mult = np.stack([_phasors(s, f, [(case["phase_l"], case["phase_m"])])[0] / s["g0"][c]
                     for c, f in enumerate(s["freqs"])])
    mult = torch.as_tensor(mult, device="cuda")
    for c, f in enumerate(s["freqs"]):
        e = _exact_volt(case, s, volt, c)
        pix = []
        for t in range(0, T, step):
            x = _fields(case, taps[c], e[t:t + step] * mult[c])
            image[c] += (x.real ** 2 + x.imag ** 2).sum(0) / T
            pix.append(x[:, n // 2, n // 2].clone())
        if case["kind"] != "grad":
            gains[c] = _exact_gains(case, s, f, c, taps[c], e, torch.cat(pix))
    if case["kind"] != "grad":
        return {"image": image, "gains": torch.as_tensor(gains)}
    # dL/dI = 2 (I - M); 2 dL/dconj(w) = (2 / T) sum_t conj(E_a) sum_j W_a(j) [F^H 2 (I - M) X]_j
    r = 2 * (image - _model_image(case, s, taps))
    grad = torch.empty((nc, na), dtype=torch.complex128, device="cuda")
    for c in range(nc):
        e = _exact_volt(case, s, volt, c)
        idx, w = taps[c]
        acc = torch.zeros(na, dtype=torch.complex128, device="cuda")
        for t in range(0, T, step):
            x = _fields(case, taps[c], e[t:t + step] * mult[c]) * r[c]
            y = torch.fft.fftshift(torch.fft.fft2(torch.fft.ifftshift(x, dim=(1, 2))), dim=(1, 2)).reshape(-1, n * n)
            for j in range(idx.shape[1]):
                acc += (e[t:t + step].conj() * y[:, idx[:, j]]).sum(0) * w[:, j]
        grad[c] = 2 * acc / (T * na)
    g = torch.as_tensor(s["g0"], device="cuda")
    return {"image": image, "grad": grad * (-1 / g ** 2).conj()}
