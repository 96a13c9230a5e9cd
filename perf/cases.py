"""Performance cases: the calls a user of the library makes, over the sizes it is used at.

One ensemble of row-column-array channel data goes through beamforming into projection planes, localisation, and
the steps around them (motion estimation, SVD clutter filter, speed separation, the learned localiser); several
small ensembles go through the batch plan.  Geometries are the library's "tiny" (32 + 32 elements, 80 x 32 planes)
and "paper" (128 + 128 elements, 250 x 128 planes, 300 frames) workloads and odd sizes between them.

Inputs are drawn on the GPU from the seed: channel data of point scatterers (moving microbubbles over tissue 40 dB
brighter, 30 dB noise), planes of moving Gaussian blobs whose phase follows their axial speed, slices of a
moving speckle field or of low-rank tissue over blood.  `exact` restates each path in 64 bits with torch alone.
"""
import math
import random
from types import SimpleNamespace

import numpy as np
import torch

from paper_2511_21647_gb300 import _lib as L
from paper_2511_21647_gb300 import rca as R
from paper_2511_21647_gb300.pipeline import RcaSession

DEV = "cuda"
C32, C16F, C16BF = L.RCA_C32, L.RCA_C16F, L.RCA_C16BF
RF = {"f32": L.RCA_F32, "f16": L.RCA_F16, "i16": L.RCA_I16}
CPX = {"c32": C32, "c16f": C16F, "c16bf": C16BF}
REAL = {"c32": torch.float32, "c16f": torch.float16, "c16bf": torch.bfloat16}
SIZE = {"f32": 4, "f16": 2, "i16": 2, "c32": 8, "c16f": 4, "c16bf": 4}
PRF = 400.0
FIR_HALF = 15
CNN_LAYERS = ((1, 32), (32, 32), (32, 32), (32, 16))
#: slow-time lengths of the separation (prime factors 2, 3 and 5)
SEP_FRAMES = (60, 64, 72, 80, 90, 96, 100, 120, 125, 128, 144, 150, 160, 180, 192, 200, 216, 240, 243, 250, 256, 288, 300)


# --- the cases -------------------------------------------------------------------------------------------------------

def _tiny(**kw):
    return dict(n_el=32, P=8, K=1, nz=80, ns=256, z0_mm=5.0, **kw)


def _paper(**kw):
    return dict(n_el=128, P=8, K=4, nz=250, ns=1024, z0_mm=20.0, **kw)


def listed():
    return [
        # the smallest call: a short acquisition of the tiny array, beamformed by one call (latency, launches)
        dict(name="beamform-tiny", kind="beamform", **_tiny(frames=8, n_mb=20, rf="f32", iq="c32", planes="c32")),
        # a mid-size array with an odd record, half-precision channel data and odd plane rows
        dict(name="beamform-ragged", kind="beamform", n_el=96, P=8, K=3, nz=187, ns=771, z0_mm=12.0, frames=45, n_mb=100,
             rf="f16", iq="c32", planes="c32"),
        # the paper's ensemble in full precision: the library's headline call
        dict(name="beamform-paper", kind="beamform", **_paper(frames=300, n_mb=200, rf="f32", iq="c32", planes="c32")),
        # the same ensemble in the reduced precision form: int16 channel data, FP16 IQ, BF16 planes
        dict(name="beamform-paper-i16", kind="beamform",
             **_paper(frames=300, n_mb=200, rf="i16", iq="c16f", planes="c16bf")),
        # sixteen uneven small ensembles (100 to 600 frames, 2 to 8 transmissions) as one captured batch
        dict(name="batch-16", kind="batch", n=16, f_min=100, f_max=600, mix=4000),
        # localisation of a tiny ensemble: short lists, many small launches
        dict(name="localize-tiny", kind="localize", d=5, planes="c32", **_tiny(frames=64, n_mb=20)),
        # localisation of the paper's ensemble (enhancement, 11 x 11 NCC, peaks, pairing)
        dict(name="localize-paper", kind="localize", d=11, planes="c32", **_paper(frames=300, n_mb=500)),
        # rigid motion of every frame of the paper's ensemble from its unfiltered slices
        dict(name="motion-paper", kind="motion", **_paper(frames=300)),
        # eigen-based clutter filter of the same slices (kept unfiltered for the motion, so a copy is filtered)
        dict(name="svd-paper", kind="svd", rank=16, **_paper(frames=300)),
        # three speed bands x two directions of the paper's planes, each with its enhancement
        dict(name="separate-paper", kind="separate", bands=3, planes="c32", **_paper(frames=300, n_mb=500)),
        # learned localiser: heatmaps of 16 frames of the paper's planes (the chunk a caller keeps on the device)
        dict(name="infer-paper", kind="infer", **_paper(frames=16, n_mb=500)),
        # learned localiser: one training step of 64 planes of the tiny geometry
        dict(name="train-tiny", kind="train", batch=64, H=80, W=32),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("beamform", "beamform", "beamform", "localize", "localize", "motion", "svd", "separate", "infer",
                       "train", "batch"))
    if kind == "batch":
        return dict(kind=kind, n=rng.randint(2, 16), f_min=rng.randint(20, 100), f_max=rng.randint(101, 600),
                    mix=rng.randrange(1 << 20))
    if kind == "train":
        return dict(kind=kind, batch=_log(rng, 8, 64), H=rng.randint(40, 120), W=rng.choice((32, 40, 48, 64)))
    n_el = rng.choice((32, 64, 128)) if kind == "motion" else rng.choice((32, 48, 64, 72, 96, 104, 128))
    nz = rng.randint(60, 250)
    c = dict(kind=kind, n_el=n_el, P=8, K=rng.randint(1, 4), nz=nz, ns=int(4.06 * nz) + rng.randint(9, 60),
             z0_mm=round(rng.uniform(5.0, 20.0), 2))
    c["frames"] = _log(rng, 8, 300)
    if kind == "beamform":
        rf, iq, planes = rng.choice((("f32", "c32", "c32"), ("f32", "c32", "c32"), ("f16", "c32", "c32"),
                                     ("i16", "c16f", "c16bf"), ("i16", "c16f", "c16f"), ("i16", "c16bf", "c16bf")))
        return dict(c, n_mb=rng.randint(10, 100), rf=rf, iq=iq, planes=planes)
    if kind == "localize":
        return dict(c, n_mb=rng.randint(2, 4) * n_el, d=rng.choice((5, 7, 9, 11)), planes=rng.choice(("c32", "c16bf")))
    if kind == "motion":
        return c
    if kind == "svd":
        c["frames"] = _log(rng, 40, 300)
        return dict(c, rank=rng.randint(2, 20))
    if kind == "separate":
        c["frames"] = rng.choice(SEP_FRAMES)
        return dict(c, n_mb=2 * n_el, bands=rng.randint(1, 3), planes=rng.choice(("c32", "c16bf")))
    c["frames"] = rng.randint(1, 16)
    return dict(c, n_mb=2 * n_el)


# --- geometry --------------------------------------------------------------------------------------------------------

def _angles(K):
    """steering angles of the RC and CR transmissions: +3 / -3 degrees for one each, else evenly over +-3 degrees"""
    if K == 1:
        return (math.radians(3.0),), (math.radians(-3.0),)
    a = tuple(math.radians(-3.0 + 6.0 * j / (K - 1)) for j in range(K))
    return a, a


def _geom(c):
    rc, cr = _angles(c["K"])
    g = SimpleNamespace(n_el=c["n_el"], P=c["P"], K=c["K"], nz=c["nz"], ns=c["ns"], us=2, pitch=0.214e-3, fc=7.8e6,
                        fs=31.2e6, c=1540.0, z0=c["z0_mm"] * 1e-3, dz=0.1e-3, fnum=1.0, ang_rc=rc, ang_cr=cr)
    g.nzs = (g.nz - 1) * g.us + 1
    g.S = g.n_el // g.P
    return g


def _batch_parts(c):
    """the ensembles of a batch: tiny geometry, uneven frame counts, 2, 4 or 8 transmissions"""
    r = random.Random(c["mix"])
    return [dict(_tiny(frames=r.randint(c["f_min"], c["f_max"]), n_mb=20, rf="f32", iq="c32", planes="c32"),
                 K=r.choice((1, 2, 4))) for _ in range(c["n"])]


# --- inputs ----------------------------------------------------------------------------------------------------------

def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _bubbles(c, g, rng):
    """positions [F][n_mb][3] (metres) and amplitudes of bubbles moving at 5 to 20 mm/s; axial speed (m/s)"""
    n, F = c["n_mb"], c["frames"]
    half = 0.5 * g.n_el * g.pitch
    lo, size = np.array([-half, -half, g.z0]), np.array([2 * half, 2 * half, g.nz * g.dz])
    v = rng.standard_normal((n, 3))
    v *= rng.uniform(5e-3, 20e-3, (n, 1)) / np.linalg.norm(v, axis=1, keepdims=True)
    t = np.arange(F)[:, None, None] / PRF
    pos = lo + np.mod(rng.random((n, 3)) * size + v * t, size)
    return pos, 10.0 ** (rng.uniform(-5, 5, n) / 20.0), v[:, 2]


def _echoes(g, pos, amp):
    """[F][2K][E][ns] channel data of scatterers pos [F][n][3]: complex spikes of whole-number weight at the nearest
    sample (so that the sum does not depend on its order), carrying the phase of the rest of the delay, convolved
    with the 65 % bandwidth pulse."""
    p = torch.as_tensor(pos, device=DEV, dtype=torch.float64)
    a = torch.as_tensor(amp, device=DEV, dtype=torch.float64)
    F, n, _ = p.shape
    E, ns = g.n_el, g.ns
    u = (torch.arange(E, device=DEV, dtype=torch.float64) - 0.5 * (E - 1)) * g.pitch
    sig = math.sqrt(2 * math.log(2)) / (math.pi * 0.65 * g.fc) * g.fs
    m = torch.arange(-8, 9, device=DEV, dtype=torch.float64)
    pulse = (torch.exp(-m * m / (2 * sig * sig)) * torch.exp(2j * math.pi * g.fc / g.fs * m)).to(torch.complex64)
    nfft = 1 << (ns + 40 - 1).bit_length()
    spec = torch.fft.fft(pulse, n=nfft)
    out = torch.empty((F, 2 * g.K, E, ns), device=DEV, dtype=torch.float32)
    step = max(1, (1 << 24) // (n * E))
    base = torch.arange(E, device=DEV)[None, :, None] * nfft
    for f0 in range(0, F, step):
        q = p[f0:f0 + step]
        for k, th in enumerate(g.ang_rc + g.ang_cr):
            trans, recv = (q[..., 1], q[..., 0]) if k < g.K else (q[..., 0], q[..., 1])
            z = q[..., 2]
            tx = (z * math.cos(th) + trans * math.sin(th) + 0.5 * E * g.pitch * abs(math.sin(th))) / g.c
            rx = torch.sqrt((recv[:, None, :] - u[None, :, None]) ** 2 + z[:, None, :] ** 2) / g.c
            s = (tx[:, None, :] + rx - 2 * g.z0 / g.c) * g.fs + 8.0
            near = torch.round(s)
            w = 4096.0 * a * torch.exp(2j * math.pi * g.fc / g.fs * (near - s))
            ok = (near >= 0) & (near < ns + 16)
            w = torch.where(ok, w, torch.zeros((), device=DEV, dtype=w.dtype))
            at = (torch.arange(q.shape[0], device=DEV)[:, None, None] * E * nfft + base
                  + torch.where(ok, near, torch.zeros((), device=DEV, dtype=near.dtype)).long()).reshape(-1)
            parts = []
            for x in (w.real, w.imag):
                acc = torch.zeros(q.shape[0] * E * nfft, device=DEV, dtype=torch.float32)
                parts.append(acc.index_add_(0, at, torch.round(x).float().reshape(-1)))
            spikes = torch.complex(*parts).view(q.shape[0], E, nfft)
            y = torch.fft.ifft(torch.fft.fft(spikes) * spec)
            out[f0:f0 + step, k] = y.real[..., 16:16 + ns] / 4096.0
    return out


def _channel_data(c, g, seed):
    """[F][2K][E][ns] float: moving bubbles, tissue 40 dB brighter that sways a little, noise 30 dB below the bubbles"""
    rng = np.random.Generator(np.random.PCG64(seed))
    pos, amp, _ = _bubbles(c, g, rng)
    rf = _echoes(g, pos, amp)
    gen = _gen(seed)
    noise = float(rf.square().mean().sqrt()) * 10.0 ** (-30 / 20)
    half = 0.5 * g.n_el * g.pitch
    lo, size = np.array([-half, -half, g.z0]), np.array([2 * half, 2 * half, g.nz * g.dz])
    t_pos, t_amp = lo + rng.random((2, 300, 3)) * size, 100.0 * rng.choice([-1.0, 1.0], 300)
    still, sway = _echoes(g, t_pos, t_amp)
    s = 0.01 * torch.sin(2 * math.pi * torch.arange(c["frames"], device=DEV) / PRF)
    for f in range(c["frames"]):
        rf[f].add_(still).add_(sway * s[f])
        rf[f].add_(torch.randn(rf[f].shape, generator=gen, device=DEV), alpha=noise)
    return rf


def _rf_typed(c, g, seed):
    """channel data in the case's type: (rf, scale or None)"""
    rf = _channel_data(c, g, seed)
    if c["rf"] == "i16":
        scale = (rf.abs().amax(dim=(0, 3)) / 32767.0).clamp_(min=1e-30)
        return torch.round(rf / scale[None, :, :, None]).clamp_(-32767, 32767).to(torch.int16), scale
    return (rf.half() if c["rf"] == "f16" else rf), None


def _planes(c, g, seed, sig_z=0.81, sig_lat=1.45):
    """[F][2][2][S][nz][N][2]: moving blobs (RC and CR alike), their phase following the axial speed, a weak still
    background and noise of each plane's own"""
    rng = np.random.Generator(np.random.PCG64(seed))
    gen = _gen(seed)
    F, S, N, nz = c["frames"], g.S, g.n_el, g.nz
    pos, amp, vz = _bubbles(c, g, rng)
    px = torch.as_tensor((pos - np.array([0, 0, g.z0])) / np.array([g.pitch, g.pitch, g.dz])
                         + np.array([0.5 * (N - 1), 0.5 * (N - 1), 0]), device=DEV, dtype=torch.float32)
    t = np.arange(F)[:, None] / PRF
    ph = rng.uniform(0, 2 * math.pi, c["n_mb"]) - 4 * math.pi * g.fc * vz * t / g.c
    w = torch.as_tensor(10.0 * amp * np.exp(1j * ph), device=DEV).to(torch.complex64)
    out = torch.empty((F, 2, 2, S, nz, N, 2), device=DEV, dtype=REAL[c.get("planes", "c32")])
    still = 0.3 * torch.randn((2, 2, S, nz, N, 2), generator=gen, device=DEV)
    zz = torch.arange(nz, device=DEV, dtype=torch.float32)
    xx = torch.arange(N, device=DEV, dtype=torch.float32)
    step = max(1, (1 << 26) // (S * nz * c["n_mb"]))
    for f0 in range(0, F, step):
        q, wq = px[f0:f0 + step], w[f0:f0 + step]
        gz = torch.exp(-(zz - q[..., 2, None]) ** 2 / (2 * sig_z ** 2))                       # [T][n][nz]
        for axis in range(2):
            lat, tr = q[..., axis], q[..., 1 - axis]
            gl = torch.exp(-(xx - lat[..., None]) ** 2 / (2 * sig_lat ** 2))                  # [T][n][N]
            slab = torch.div(tr.round(), g.P, rounding_mode="floor").clamp(0, S - 1)
            member = (slab[:, None, :] == torch.arange(S, device=DEV)[None, :, None]).float()  # [T][S][n]
            for part, x in enumerate((wq.real, wq.imag)):
                a = (member * x[:, None, :])[:, :, None, :] * gz.transpose(1, 2)[:, None]      # [T][S][nz][n]
                f = a @ gl[:, None]
                for fam in range(2):
                    e = torch.randn(f.shape, generator=gen, device=DEV)
                    out[f0:f0 + step, axis, fam, ..., part] = f + still[axis, fam, ..., part] + 0.1 * e
    return out


def _moving_slices(c, g, seed):
    """[F][2K][nzs][N][2]: a smooth speckle field per transmission, displaced rigidly frame by frame, 5 % noise"""
    gen = _gen(seed)
    nt, F, Z, N = 2 * g.K, c["frames"], g.nzs, g.n_el
    kz = torch.fft.fftfreq(Z, device=DEV, dtype=torch.float64)[:, None]
    kx = torch.fft.fftfreq(N, device=DEV, dtype=torch.float64)[None, :]
    field = torch.randn((nt, Z, N), generator=gen, device=DEV, dtype=torch.complex64)
    spec = torch.fft.fft2(field) * torch.exp(-2 * math.pi ** 2 * ((2.0 * kz) ** 2 + kx ** 2)).float()
    spec = spec * (Z * N) ** 0.5 / spec.abs().square().mean().sqrt()
    a = 2 * math.pi * torch.rand(4, generator=gen, device=DEV, dtype=torch.float64)
    out = torch.empty((F, nt, Z, N, 2), device=DEV, dtype=torch.float32)
    fam = torch.arange(nt, device=DEV) >= g.K
    for f in range(F):
        ph = 2 * math.pi * f / PRF
        dz = 4.0 * (torch.sin(ph + a[0]) - torch.sin(a[0]))
        dx = torch.where(fam, 0.8 * (torch.sin(2 * ph + a[1]) - torch.sin(a[1])),
                         0.8 * (torch.sin(3 * ph + a[2]) - torch.sin(a[2])))
        shift = torch.exp(-2j * math.pi * (kz * dz + kx * dx[:, None, None])).to(torch.complex64)
        s = torch.fft.ifft2(spec * shift) / (Z * N) ** -0.5
        out[f] = torch.view_as_real(s / s.abs().square().mean().sqrt())
        out[f].add_(torch.randn(out[f].shape, generator=gen, device=DEV), alpha=0.05)
    return out


def _tissue_slices(c, g, seed):
    """[F][2K][nzs][N][2]: `rank` tissue components of falling strength, 26 dB above the blood and noise together"""
    rng = np.random.Generator(np.random.PCG64(seed))
    gen = _gen(seed)
    nt, F, n, r = 2 * g.K, c["frames"], g.nzs * g.n_el, c["rank"]
    out = torch.empty((F, nt, n, 2), device=DEV, dtype=torch.float32)
    s = torch.as_tensor(np.geomspace(1.0, 0.2, r), device=DEV, dtype=torch.float32)
    for k in range(nt):
        v = np.linalg.qr(rng.standard_normal((F, r)) + 1j * rng.standard_normal((F, r)))[0] * math.sqrt(F)
        u = torch.randn((r, n), generator=gen, device=DEV, dtype=torch.complex64) * s[:, None]
        x = torch.as_tensor(v, device=DEV).to(torch.complex64) @ u
        x = x * (20.0 / float(x.abs().square().mean().sqrt()))
        out[:, k] = torch.view_as_real(x + torch.randn((F, n), generator=gen, device=DEV, dtype=torch.complex64))
    return out.view(F, nt, g.nzs, g.n_el, 2)


def _amplitude(c, g, seed):
    """enhanced planes A [F][2][S][nz][N] and their frame maxima M [F]"""
    p = torch.view_as_complex(_planes(c, g, seed))
    A = (p[:, :, 0] * p[:, :, 1].conj()).abs().sqrt().contiguous()
    return A, A.amax(dim=(1, 2, 3, 4))


def _cnn_params(seed):
    """He-normal weights [Cout][9][Cin] and small biases of the four layers, one flat vector"""
    rng = np.random.Generator(np.random.PCG64(seed + 77))
    flat = []
    for cin, cout in CNN_LAYERS:
        flat.append(rng.standard_normal((cout, 9, cin)) * math.sqrt(2.0 / (9 * cin)))
        flat.append(0.05 * rng.standard_normal(cout))
    return np.concatenate([x.reshape(-1) for x in flat]).astype(np.float32)


def _training_batch(c, seed):
    """A [B][H][W] (blobs over noise, largest value 1), target [B][4H][4W] (unit Gaussians)"""
    rng = np.random.Generator(np.random.PCG64(seed))
    gen = _gen(seed)
    B, H, W = c["batch"], c["H"], c["W"]
    n = 8
    z = torch.as_tensor(rng.uniform(0, H - 1, (B, n)), device=DEV, dtype=torch.float32)
    x = torch.as_tensor(rng.uniform(0, W - 1, (B, n)), device=DEV, dtype=torch.float32)
    a = torch.as_tensor(10.0 ** (rng.uniform(-5, 5, (B, n)) / 20.0), device=DEV, dtype=torch.float32)

    def blobs(h, w, zc, xc, amp, sz, sx):
        gz = torch.exp(-(torch.arange(h, device=DEV) - zc[..., None]) ** 2 / (2 * sz * sz)) * amp[..., None]
        gx = torch.exp(-(torch.arange(w, device=DEV) - xc[..., None]) ** 2 / (2 * sx * sx))
        return gz.transpose(1, 2) @ gx

    A = blobs(H, W, z, x, a, 0.81, 1.45) + 0.05 * torch.rand((B, H, W), generator=gen, device=DEV)
    T = blobs(4 * H, 4 * W, 4 * z + 1.5, 4 * x + 1.5, torch.ones_like(a), 1.0, 1.0)
    return (A / A.amax(dim=(1, 2), keepdim=True)).contiguous(), T.contiguous()


# --- what a program has in hand before the call, and the call ----------------------------------------------------------

class State:
    """a case's buffers and handles; the handles are freed with it"""

    def __init__(self, **kw):
        self.closers = []
        self.__dict__.update(kw)

    def __del__(self):
        for close in self.closers:
            close()


def _lists(bufs):
    """the integer and the float fields of the 2D and 3D lists, and their lengths (views of the buffers)"""
    o2, n2, o3, n3 = bufs
    return {"n2d": n2, "loc2d_int": o2[:, :5], "loc2d": o2.view(torch.float32)[:, 5:9],
            "n3d": n3, "loc3d_int": o3[:, :3], "loc3d": o3.view(torch.float32)[:, 4:9]}


def _ulm_params(c):
    return R.make_ulm_params(d=c["d"], sig_z=0.81, sig_lat=1.45, alpha=0.1, ncc_min=0.5)


def prepare(case, seed):
    c = case
    s = State(c=c)
    if c["kind"] == "train":
        s.h = R.rca_create(0)
        R.rca_set_stream(s.h, torch.cuda.current_stream())
        s.net = R.ulm_cnn_create(s.h, max_pixels=c["batch"] * c["H"] * c["W"])
        s.closers = [lambda n=s.net: R.ulm_cnn_destroy(n), lambda h=s.h: R.rca_destroy(h)]
        R.ulm_cnn_set_params(s.net, _cnn_params(seed))
        s.A, s.T = _training_batch(c, seed)
        s.loss = torch.zeros(1, device=DEV)
        return s
    if c["kind"] == "batch":
        s.h = R.rca_create(0)
        R.rca_set_stream(s.h, torch.cuda.current_stream())
        s.items, tables = [], {}
        for q, p in enumerate(_batch_parts(c)):
            g = _geom(p)
            if p["K"] not in tables:
                gh = R.rca_geometry_create(s.h, g)
                t = tables[p["K"]] = R.rca_delay_tables(s.h, gh)
                s.closers += [lambda t=t: R.rca_tables_destroy(t), lambda gh=gh: R.rca_geometry_destroy(gh)]
            planes = torch.empty((p["frames"], 2, 2, g.S, g.nz, g.n_el, 2), device=DEV)
            s.items.append(dict(tables=tables[p["K"]], rf=_channel_data(p, g, seed + 1000 * q), n_frames=p["frames"],
                                planes=planes))
        s.batch = R.rca_batch_create(s.h, s.items, L.RCA_F32, C32, C32)
        R.rca_batch_set_mode(s.batch, L.RCA_BATCH_STAGED)
        s.closers = [lambda b=s.batch: R.rca_batch_destroy(b)] + s.closers + [lambda h=s.h: R.rca_destroy(h)]
        s.out = [it["planes"] for it in s.items]
        return s
    g = _geom(c)
    s.sess = RcaSession(g)
    s.closers = [s.sess.close]
    F, kind = c["frames"], c["kind"]
    if kind == "beamform":
        s.rf, s.scale = _rf_typed(c, g, seed)
        s.planes = torch.empty((*s.sess.planes_shape(F), 2), dtype=REAL[c["planes"]], device=DEV)
    elif kind == "localize":
        s.planes, s.prm = _planes(c, g, seed), _ulm_params(c)
        s.cap2d = min(1 << 22, max(1 << 12, 256 * F * 2 * g.S))
        s.cap3d = min(1 << 19, max(1 << 12, 64 * F * g.S))
        s.bufs = s.sess.loc_buffers(s.cap2d, s.cap3d)
        s.out = _lists(s.bufs)
    elif kind == "motion":
        s.slices = _moving_slices(c, g, seed)
        s.motion = torch.empty((F, 3), device=DEV)
        s.shifts = torch.empty((F, 2 * g.K, 3), device=DEV)
        s.peaks = torch.empty((F, 2 * g.K, 2), dtype=torch.int32, device=DEV)
    elif kind == "svd":
        s.slices = _tissue_slices(c, g, seed)
        s.filtered = torch.empty_like(s.slices)
    elif kind == "separate":
        s.planes, s.prm = _planes(c, g, seed), R.make_sep_params(PRF, c["bands"])
        s.A = torch.empty((2 * c["bands"], *s.sess.a_shape(F)), device=DEV)
        s.M = torch.empty((2 * c["bands"], F), device=DEV)
    else:
        s.A, s.M = _amplitude(c, g, seed)
        B = F * 2 * g.S
        s.net = R.ulm_cnn_create(s.sess.h, max_pixels=B * g.nz * g.n_el)
        s.closers = [lambda n=s.net: R.ulm_cnn_destroy(n), s.sess.close]
        R.ulm_cnn_set_params(s.net, _cnn_params(seed))
        s.dims = (2 * g.S, B, g.nz, g.n_el)
        s.heat = torch.empty((B, 4 * g.nz, 4 * g.n_el), device=DEV)
    return s


def run(s):
    c = s.c
    kind = c["kind"]
    if kind == "beamform":
        return s.sess.beamform(s.rf, RF[c["rf"]], s.scale, iq_dtype=CPX[c["iq"]], planes_dtype=CPX[c["planes"]],
                               out=s.planes)
    if kind == "batch":
        R.rca_batch_run(s.batch, True, s.h)
        return s.out
    if kind == "localize":
        s.sess.localize(s.planes, s.prm, CPX[c["planes"]], s.cap2d, s.cap3d, s.bufs)
        return s.out
    if kind == "motion":
        R.rca_motion_estimate(s.sess.h, s.sess.t, s.slices, c["frames"], s.motion, s.shifts, s.peaks)
        return {"motion": s.motion, "shifts": s.shifts, "peaks": s.peaks}
    if kind == "svd":
        s.filtered.copy_(s.slices)
        R.rca_clutter_svd(s.sess.h, s.sess.t, s.filtered, c["frames"], c["rank"])
        return s.filtered
    if kind == "separate":
        R.ulm_separate_enhance(s.sess.h, s.sess.t, s.planes, CPX[c["planes"]], c["frames"], s.prm, L.ULM_ENH_XDOPPLER,
                               s.A, s.M)
        return {"A": s.A, "M": s.M}
    if kind == "infer":
        R.ulm_cnn_infer(s.net, s.A, s.M, *s.dims, s.heat)
        return s.heat
    R.ulm_cnn_train_step(s.net, s.A, None, 1, c["batch"], c["H"], c["W"], s.T, s.loss, True)
    return {"loss": s.loss, "grads": R.ulm_cnn_get_grads(s.net)}


# --- work --------------------------------------------------------------------------------------------------------------

def _beamform_work(c):
    """bytes: channel data in, planes out.  flops: 14 per (pixel, element) term of Stage 1 (an interpolated complex
    sample, a complex multiply-add), 16 per element sample and tap pair of the half-band low-pass, and 8 per
    (pixel, transmission) of the slab sums, each slab sample interpolated once"""
    g = _geom(c)
    F, nt = c["frames"], 2 * c["K"]
    rf = F * nt * g.n_el * g.ns
    planes = F * 4 * g.S * g.nz * g.n_el
    d = np.arange(g.n_el)
    terms = 0
    for r in range(g.nzs):
        z = g.z0 + r * g.dz / g.us
        inside = d[d * g.pitch <= 0.5 * z / g.fnum]
        terms += int(np.where(inside == 0, g.n_el, 2 * (g.n_el - inside)).sum())
    return {"bytes": rf * SIZE[c["rf"]] + planes * SIZE[c["planes"]],
            "flops": 14.0 * F * nt * terms + 50.0 * rf + 8.0 * c["K"] * planes * 2}


def work(case):
    c = case
    if c["kind"] == "beamform":
        return _beamform_work(c)
    if c["kind"] == "batch":
        parts = [_beamform_work(p) for p in _batch_parts(c)]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    per_px = sum(2.0 * 9 * cin * cout for cin, cout in CNN_LAYERS)
    if c["kind"] == "train":
        px = c["batch"] * c["H"] * c["W"]
        n = sum(9 * cin * cout + cout for cin, cout in CNN_LAYERS)
        return {"bytes": px * (4 + 64) + 4 * 6 * n, "flops": 3.0 * px * per_px}
    g = _geom(c)
    F, nt = c["frames"], 2 * c["K"]
    px = F * 2 * g.S * g.nz * g.n_el               # amplitude pixels; the planes hold two complex values for each
    slices = F * nt * g.nzs * g.n_el
    if c["kind"] == "localize":
        return {"bytes": 2 * px * SIZE[c["planes"]], "flops": px * (26.0 + 8 * c["d"])}
    if c["kind"] == "motion":
        zp = 1 << (g.nzs - 1).bit_length()
        pts = zp * g.n_el
        return {"bytes": slices * 8, "flops": (F * nt) * (10.0 * pts * math.log2(pts) + 8 * pts)}
    if c["kind"] == "svd":
        n = nt * g.nzs * g.n_el
        return {"bytes": 2 * slices * 8, "flops": n * (4.0 * F * F + 16.0 * F * c["rank"])}
    if c["kind"] == "separate":
        n = 2 * c["bands"]
        return {"bytes": 2 * px * SIZE[c["planes"]] + n * px * 4,
                "flops": 2 * px * (1 + n) * 5.0 * math.log2(F) + n * px * 20.0}
    return {"bytes": px * (4 + 64), "flops": px * per_px}


# --- the same in 64 bits -------------------------------------------------------------------------------------------------

def _exact_planes(c, g, rf, scale):
    """planes [F][2][2][S][nz][N][2] of channel data: mean removal, demodulation, Stage 1, Stage 2, slab sums"""
    f64, c128 = torch.float64, torch.complex128
    F, nt, E, ns = rf.shape
    N, Z, K = g.n_el, g.nzs, g.K
    full = lambda x: x.to(f64) if scale is None else x.to(f64) * scale.to(f64)[:, :, None]  # noqa: E731
    mean = torch.zeros((nt, E, ns), device=DEV, dtype=f64)
    for f in range(F):
        mean += full(rf[f])
    mean /= F
    # half-band low-pass, 31 taps
    m = np.arange(-FIR_HALF, FIR_HALF + 1)
    odd = (np.abs(m) % 2) == 1
    x = np.where(m == 0, 1.0, 0.5 * np.pi * m)
    h = np.where(odd, 0.5 * np.sin(x) / x * (0.54 + 0.46 * np.cos(np.pi * m / FIR_HALF)), 0.0)
    h *= 0.5 / h.sum()
    h[FIR_HALF] = 0.5
    t0 = 2 * g.z0 / g.c
    n = torch.arange(ns, device=DEV, dtype=f64)
    mix = torch.exp(-2j * math.pi * g.fc * (t0 + n / g.fs))
    ang = g.ang_rc + g.ang_cr
    z = g.z0 + torch.arange(Z, device=DEV, dtype=f64) * (g.dz / g.us)
    Lap = E * g.pitch
    tx = torch.stack([(z * math.cos(a) + 0.5 * Lap * abs(math.sin(a))) / g.c for a in ang])     # [nt][Z]
    row = torch.arange(g.nz, device=DEV, dtype=f64)
    u = (torch.arange(N, device=DEV, dtype=f64) - 0.5 * (N - 1)) * g.pitch
    out = torch.empty((F, 2, 2, g.S, g.nz, N, 2), device=DEV, dtype=f64)
    step = max(1, (1 << 24) // (nt * ns * E))
    for f0 in range(0, F, step):
        b = torch.stack([(full(rf[f]) - mean) * mix for f in range(f0, min(F, f0 + step))])      # [T][nt][E][ns]
        iq = torch.zeros_like(b)
        for q, w in zip(m, h):
            if w:
                lo, hi = max(0, q), min(ns, ns + q)
                if lo < hi:
                    iq[..., lo:hi] += 2 * w * b[..., lo - q:hi - q]
        iq = iq.transpose(2, 3).contiguous()                                                    # [T][nt][ns][E]
        T = iq.shape[0]
        sl = torch.zeros((T, nt, Z, N), device=DEV, dtype=c128)
        for d in range(N):
            off = d * g.pitch
            ap = z / g.fnum
            w = torch.where(off <= 0.5 * ap, torch.cos(math.pi * off / ap) ** 2, torch.zeros_like(ap))
            if not bool((w > 0).any()):
                continue
            rx = torch.sqrt(off * off + z * z) / g.c
            xi = (tx + rx - t0) * g.fs                                                          # [nt][Z]
            ok = (xi >= 0) & (xi <= ns - 1)
            n0 = xi.floor().clamp(0, ns - 1).long()
            fr = (xi - n0) * ok
            n1 = (n0 + 1).clamp(max=ns - 1)
            cw = (w * torch.exp(2j * math.pi * g.fc * (rx - z / g.c)))[None] * ok
            k = torch.arange(nt, device=DEV)[:, None]
            v = iq[:, k, n0] * (cw * (1 - fr))[None, :, :, None] + iq[:, k, n1] * (cw * fr)[None, :, :, None]
            sl[..., d:] += v[..., :N - d]
            if d:
                sl[..., :N - d] += v[..., d:]
        for f in range(T):
            for fam in range(2):
                vol = torch.zeros((g.nz, N, N), device=DEV, dtype=c128)                         # [i][u][l]
                for k in range(fam * K, fam * K + K):
                    a = ang[k]
                    sh = u * math.sin(a) / (1 + math.cos(a))
                    zeta = g.us * row[:, None] + sh[None, :] * g.us / g.dz
                    ok = (zeta >= 0) & (zeta <= Z - 1)
                    n0 = zeta.floor().clamp(0, Z - 1).long()
                    fr = (zeta - n0) * ok
                    n1 = (n0 + 1).clamp(max=Z - 1)
                    tau = ((g.z0 + row[:, None] * g.dz + sh) * (1 + math.cos(a)) + 0.5 * Lap * abs(math.sin(a))) / g.c
                    car = torch.exp(2j * math.pi * g.fc * tau) * ok
                    vol += sl[f, k][n0] * (car * (1 - fr))[..., None] + sl[f, k][n1] * (car * fr)[..., None]
                across = vol.view(g.nz, g.S, g.P, N).sum(2).transpose(0, 1)                     # [S over u][i][l]
                along = vol.view(g.nz, N, g.S, g.P).sum(3).permute(2, 0, 1)                     # [S over l][i][u]
                # RC slices resolve x (XZ: slab over y), CR slices y (YZ: slab over x)
                out[f0 + f, fam, fam] = torch.view_as_real(across)
                out[f0 + f, 1 - fam, fam] = torch.view_as_real(along)
    return out


def _exact_motion(c, g, x):
    F, nt = x.shape[:2]
    zp = 1 << (g.nzs - 1).bit_length()
    ref = torch.fft.fft2(torch.view_as_complex(x[0].double()), s=(zp, g.n_el)).conj()
    shifts = torch.empty((F, nt, 3), device=DEV, dtype=torch.float64)

    def vertex(lo, mid, hi):
        den = lo - 2 * mid + hi
        return torch.where(den >= 0, torch.zeros_like(den), ((lo - hi) / (2 * den)).clamp(-0.5, 0.5))

    norm = [torch.view_as_complex(x[f].double()).abs().square().sum((1, 2)).sqrt() for f in range(F)]
    for f in range(F):
        r = torch.fft.ifft2(torch.fft.fft2(torch.view_as_complex(x[f].double()), s=(zp, g.n_el)) * ref).abs()
        at = r.view(nt, -1).argmax(1)
        iz, ix = torch.div(at, g.n_el, rounding_mode="floor"), at % g.n_el
        k = torch.arange(nt, device=DEV)
        pk = r[k, iz, ix]
        sz = vertex(r[k, (iz - 1) % zp, ix], pk, r[k, (iz + 1) % zp, ix])
        sx = vertex(r[k, iz, (ix - 1) % g.n_el], pk, r[k, iz, (ix + 1) % g.n_el])
        shifts[f, :, 0] = torch.where(iz < zp // 2, iz, iz - zp) + sz
        shifts[f, :, 1] = torch.where(ix < g.n_el // 2, ix, ix - g.n_el) + sx
        shifts[f, :, 2] = pk / (norm[f] * norm[0])
    m = shifts.view(F, 2, g.K, 3).mean(2)
    motion = torch.stack([m[:, 0, 1] * g.pitch, m[:, 1, 1] * g.pitch,
                          0.5 * (m[:, 0, 0] + m[:, 1, 0]) * g.dz / g.us], 1)
    return {"motion": motion, "shifts": shifts, "peaks": None}


def _exact_svd(c, x):
    F, nt = x.shape[:2]
    out = torch.empty(x.shape, device=DEV, dtype=torch.float64)
    for k in range(nt):
        m = torch.view_as_complex(x[:, k].double().contiguous()).reshape(F, -1)                 # rows: frames
        v = torch.linalg.eigh((m.conj() @ m.T).cpu())[1][:, -c["rank"]:].to(DEV)                # of X^H X, X = m^T
        # X - X V V^H, transposed: m - conj(V) (V^T m)
        out[:, k] = torch.view_as_real(m - v.conj() @ (v.T @ m)).view(out[:, k].shape)
    return out


def _exact_separate(c, planes):
    F, nb = c["frames"], c["bands"]
    shape = planes.shape[1:-1]                                                                  # [2][2][S][nz][N]
    A = torch.empty((2 * nb, F, shape[0], *shape[2:]), device=DEV, dtype=torch.float64)
    j = torch.arange(F, device=DEV)
    k = torch.where(2 * j < F, j, j - F)
    hz = k.abs().double() * PRF / F
    live = (k != 0) & (2 * j != F)
    near = torch.ones((F, F), device=DEV, dtype=torch.float64).triu(-1).tril(1)
    for a in range(shape[0]):
        for s in range(shape[2]):
            x = torch.fft.fft(torch.view_as_complex(planes[:, a, :, s].double().contiguous()), dim=0)  # [F][2][nz][N]
            for b in range(2 * nb):
                lo, hi = (b % nb) * PRF / (2 * nb), (b % nb + 1) * PRF / (2 * nb)
                keep = live & ((k > 0) == (b < nb)) & (hz > lo) & (hz <= hi)
                y = torch.fft.ifft(x * keep[:, None, None, None], dim=0)
                q = (y[:, 0] * y[:, 1].conj()).reshape(F, -1)
                q = torch.complex(near @ q.real, near @ q.imag)
                A[b, :, a, s] = q.abs().sqrt().view(F, *shape[3:])
    return {"A": A, "M": A.amax(dim=(2, 3, 4, 5))}


def _unflatten(flat):
    p, o = [], 0
    for cin, cout in CNN_LAYERS:
        w = flat[o:o + cout * 9 * cin].view(cout, 3, 3, cin).permute(0, 3, 1, 2)
        o += cout * 9 * cin
        p.append((w, flat[o:o + cout]))
        o += cout
    return p


def _conv(x, w, b):
    """3 x 3 convolution with zero borders as nine products [.., Cin] x [Cin, Cout]; x [B][H][W][Cin]"""
    B, H, W, _ = x.shape
    x = torch.nn.functional.pad(x, (0, 0, 1, 1, 1, 1))
    return sum(x[:, dy:dy + H, dx:dx + W] @ w[:, :, dy, dx].T for dy in range(3) for dx in range(3)) + b


def _network(x, layers):
    """x [B][H][W] -> heatmap [B][4H][4W]"""
    B, H, W = x.shape
    x = x[..., None]
    for q, (w, b) in enumerate(layers):
        x = _conv(x, w, b)
        x = torch.relu(x) if q < 3 else x
    return x.view(B, H, W, 4, 4).permute(0, 1, 3, 2, 4).reshape(B, 4 * H, 4 * W)


def exact(case, seed):
    c = case
    kind = c["kind"]
    if kind == "localize":
        return None                    # lists of decisions
    if kind == "train":
        A, T = _training_batch(c, seed)
        flat = torch.as_tensor(_cnn_params(seed), device=DEV).double().requires_grad_(True)
        loss = (_network(A.double(), _unflatten(flat)) - T.double()).square().mean()
        loss.backward()
        return {"loss": loss.detach().view(1), "grads": flat.grad}
    if kind == "batch":
        out = []
        for q, p in enumerate(_batch_parts(c)):
            g = _geom(p)
            out.append(_exact_planes(p, g, _channel_data(p, g, seed + 1000 * q), None))
        return out
    g = _geom(c)
    if kind == "beamform":
        return _exact_planes(c, g, *_rf_typed(c, g, seed))
    if kind == "motion":
        return _exact_motion(c, g, _moving_slices(c, g, seed))
    if kind == "svd":
        return _exact_svd(c, _tissue_slices(c, g, seed))
    if kind == "separate":
        return _exact_separate(c, _planes(c, g, seed))
    A, M = _amplitude(c, g, seed)
    layers = _unflatten(torch.as_tensor(_cnn_params(seed), device=DEV).double())
    x = (A / M.clamp(min=1e-30)[:, None, None, None, None]).double().view(-1, g.nz, g.n_el)
    return torch.cat([_network(x[q:q + 32], layers) for q in range(0, x.shape[0], 32)])
