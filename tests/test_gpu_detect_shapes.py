"""2D detection at the widths and kernel lengths where its block size, its compile-time variants and its candidate
list change (up to 64 columns: half the threads; a threshold that lets more pixels through than the serving warp's
list holds): the list is the peak rule's on the kernel's own NCC map, value for value (the map itself is compared
with the oracle in test_gpu_localize).  Pairing of lists of a few to many entries per plane against the oracle."""
from dataclasses import replace

import numpy as np
import pytest
import torch
from scipy.ndimage import gaussian_filter

import oracle as O

pytestmark = pytest.mark.gpu


def _peaks(A, M, ncc, alpha, ncc_min):
    """the peak rule on NCC maps (float32, the kernel's own): regional maxima over both thresholds, strict against
    earlier neighbours, in raster order, with float32 parabolas"""
    out = []
    F, _, S, nz, N = A.shape
    thr = np.float32(alpha) * M

    def vertex(lo, mid, hi):
        den = lo - np.float32(2) * mid + hi
        if den >= 0:
            return np.float32(0)
        return min(np.float32(0.5), max(np.float32(-0.5), (lo - hi) / (np.float32(2) * den)))

    for t in range(F):
        for axis in range(2):
            for b in range(S):
                n, c = ncc[t, axis, b], ncc[t, axis, b, 1:-1, 1:-1]
                ok = (c >= np.float32(ncc_min)) & (A[t, axis, b, 1:-1, 1:-1] >= thr[t])
                for di in (-1, 0, 1):
                    for dl in (-1, 0, 1):
                        if di or dl:
                            q = n[1 + di:nz - 1 + di, 1 + dl:N - 1 + dl]
                            ok &= (c > q) if di < 0 or (di == 0 and dl < 0) else (c >= q)
                for i, l in zip(*(1 + x for x in np.nonzero(ok))):
                    out.append((t, axis, b, i, l, np.float32(i) + vertex(n[i - 1, l], n[i, l], n[i + 1, l]),
                                np.float32(l) + vertex(n[i, l - 1], n[i, l], n[i, l + 1]), n[i, l], A[t, axis, b, i, l]))
    return out


@pytest.mark.parametrize("N,nz,d,ncc_min", [(32, 61, 5, 0.5), (48, 30, 3, 0.3), (64, 31, 11, 0.5), (64, 92, 7, -0.99),
                                            (72, 40, 9, 0.5), (96, 59, 15, 0.4), (104, 33, 11, -0.99), (128, 75, 13, 0.5),
                                            (128, 64, 11, -0.99), (256, 45, 11, 0.5), (256, 32, 15, -0.99)])
def test_detection_sizes(tiny, N, nz, d, ncc_min):
    from paper_2511_21647_gb300 import rca
    from paper_2511_21647_gb300.pipeline import RcaSession, list2d_numpy
    g = replace(tiny.geom, n_el=N, nz=nz)
    F, S = 3, N // g.P
    rng = np.random.default_rng(N + d)
    A = rng.random((F, 2, S, nz, N))
    A = gaussian_filter(A, (0, 0, 0, 3.0, 3.0)) if ncc_min < 0 else gaussian_filter(A, (0, 0, 0, 0.9, 1.5))
    A = ((A - A.min()) ** 2).astype(np.float32)
    M = A.max(axis=(1, 2, 3, 4))
    prm = rca.make_ulm_params(d=d, sig_z=0.81, sig_lat=1.45, alpha=0.05, ncc_min=ncc_min)
    with RcaSession(g) as s:
        out, n2d, ncc = s.detect2d(torch.from_numpy(A).cuda(), torch.from_numpy(M).cuda(), prm, want_ncc=True)
        got = list2d_numpy(out, int(n2d.item()))
        assert s.sync_status() == 0
    ref = _peaks(A, M, ncc.cpu().numpy(), 0.05, ncc_min)
    assert len(ref) > 20 and len(got) == len(ref)
    # a row next to a strip of 30 rows' border is also computed in the other strip, its sums split elsewhere:
    # there the kernel's z comes from a neighbour that the map does not hold (1e-3 px, the lists' bound)
    inner = ~np.isin(got["iz"] % 30, (0, 29))
    assert np.allclose(got["z"], np.array([r[5] for r in ref]), rtol=0, atol=1e-3)
    for q, f in enumerate(("frame", "axis", "slab", "iz", "ilat", "z", "lat", "ncc", "amp")):
        w = inner if f == "z" else slice(None)
        assert np.array_equal(got[f][w], np.array([r[q] for r in ref], dtype=got[f].dtype)[w]), f


@pytest.mark.parametrize("per_plane,equal", [(1, False), (9, False), (40, False), (12, True)])
def test_pairing_sizes(tiny, per_plane, equal):
    """lists of a few to many entries per plane; equal: amplitudes of two values only, so that costs tie"""
    from paper_2511_21647_gb300 import _lib
    from paper_2511_21647_gb300.pipeline import RcaSession, list3d_numpy
    g = tiny.geom
    F, S, N = 16, g.n_el // g.P, g.n_el
    rng = np.random.default_rng(per_plane)
    rec = np.zeros(F * 2 * S * per_plane, dtype=_lib.LOC2D)
    rec["frame"] = np.repeat(np.arange(F), 2 * S * per_plane)
    rec["axis"] = np.tile(np.repeat([0, 1], S * per_plane), F)
    rec["slab"] = np.tile(np.repeat(np.arange(S), per_plane), 2 * F)
    rec["iz"], rec["ilat"] = rng.integers(1, 8, len(rec)), rng.integers(1, N - 1, len(rec))
    rec["z"] = (rec["iz"] + rng.uniform(-0.5, 0.5, len(rec))).astype(np.float32)
    rec["lat"] = rec["ilat"]
    rec["amp"] = rng.choice([1.0, 1.05], len(rec)) if equal else rng.uniform(0.9, 1.1, len(rec)).astype(np.float32)
    L_o = np.zeros(len(rec), dtype=O.LOC2D)
    for f in ("frame", "axis", "slab", "iz", "ilat", "z", "lat", "ncc", "amp"):
        L_o[f] = rec[f]
    ref = O.pair3d(L_o, g.P)
    dev = torch.from_numpy(rec.view(np.int32).reshape(-1, 10).copy()).cuda()
    n2d = torch.tensor([len(rec)], dtype=torch.int32, device="cuda")
    with RcaSession(g) as s:
        out, n3d = s.pair3d(dev, n2d, len(rec), F)
        got = list3d_numpy(out, int(n3d.item()))
        assert s.sync_status() == 0
    assert len(ref) > 0 and len(got) == len(ref)
    for f in ("frame", "i_xz", "i_yz"):
        assert np.array_equal(got[f], ref[f]), f
